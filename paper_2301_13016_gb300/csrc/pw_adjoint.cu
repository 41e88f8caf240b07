// Adjoint (transpose) of the PW scheme linearised about (u, v, w): the
// sensitivities of a scalar with respect to u, v, w given its sensitivities
// l = (lsu, lsv, lsw) with respect to the source terms (Sec. 2.2 defines the
// scheme; its transpose is what data assimilation and gradient-based
// training of the velocity fields need).
//
// Every term of the scheme has the shape c * a * (b + d) at an output cell X;
// its transpose sends c*l(X)*(b+d) to the slot of a and c*l(X)*a to the slots
// of b and d.  The kernel is written in GATHER form: one thread per input
// cell C collects, field by field, the contributions of every output X whose
// stencil touches C (up to nine per field), so no two threads write the same
// cell and no atomics are needed.  Output sensitivities outside the scheme's
// output set (levels other than 2..nz for su, sv and 2..nz-1 for sw; the
// upper vertical term only below the lid; lateral halo cells) are zero.
//
// Modes: full-array (C ranges over levels 1..nz of the interior plus the
// one-cell lateral halo; halo values of u, v, w are independent inputs), or
// periodic (C ranges over the interior; output cells wrap around the doubly
// periodic domain, which equals the full-array result folded back onto the
// interior; u, v, w must carry periodic halos).
#include <algorithm>

#include "pw_device.cuh"

#include <type_traits>
#include "pw_internal.h"

namespace pw {

struct AdjArgs {
    const float *u, *v, *w;        // linearisation point
    const float *lu, *lv, *lw;     // sensitivities to su, sv, sw
    float *gu, *gv, *gw;           // result
    float alpha;                   // g = [g or l or 0] + alpha * J^T l
    int accumulate, add_lambda, periodic;
};

// J^T l at one cell: the terms of every output whose stencil touches it, each
// skipped when its sensitivity is exactly 0 (or does not exist).
__device__ __forceinline__ void adjoint_gather_cell(const GridDev& g, const AdjArgs& a, const CoefDev& cf, const int K,
                                                    const int J, const int I, float& ru, float& rv, float& rw) {
    const int nx = g.nx, ny = g.ny, nz = g.nz, nzp2 = nz + 2;
    const float* tzc1 = cf.tz;
    const float* tzc2 = cf.tz + nzp2;
    const float* tzd1 = cf.tz + 2 * nzp2;
    const float* tzd2 = cf.tz + 3 * nzp2;
    const float tcx = cf.tcx, tcy = cf.tcy;
    auto off = [&](int k, int j, int i) { return g.origin + (long long)k * g.pk + (long long)j * g.pj + i; };
    auto U = [&](int k, int j, int i) { return __ldg(a.u + off(k, j, i)); };
    auto V = [&](int k, int j, int i) { return __ldg(a.v + off(k, j, i)); };
    auto W = [&](int k, int j, int i) { return __ldg(a.w + off(k, j, i)); };
    // output cell X = (k, j, i): is it an output of the scheme, and where
    // does its sensitivity live (wrapped in periodic mode)?
    auto out_ok = [&](int k, int j, int i, int klo, int khi, int& jj, int& ii) {
        if (k < klo || k > khi) return false;
        if (a.periodic) {
            jj = j < 1 ? j + ny : (j > ny ? j - ny : j);
            ii = i < 1 ? i + nx : (i > nx ? i - nx : i);
            return true;
        }
        jj = j;
        ii = i;
        return j >= 1 && j <= ny && i >= 1 && i <= nx;
    };
    // l at X for su (levels 2..nz), sv (2..nz), sw (2..nz-1); the upper
    // vertical terms of su, sv exist only below the lid (levels 2..nz-1)
    auto LU = [&](int k, int j, int i, int khi) {
        int jj, ii;
        return out_ok(k, j, i, 2, khi, jj, ii) ? __ldg(a.lu + off(k, jj, ii)) : 0.f;
    };
    auto LV = [&](int k, int j, int i, int khi) {
        int jj, ii;
        return out_ok(k, j, i, 2, khi, jj, ii) ? __ldg(a.lv + off(k, jj, ii)) : 0.f;
    };
    auto LW = [&](int k, int j, int i) {
        int jj, ii;
        return out_ok(k, j, i, 2, nz - 1, jj, ii) ? __ldg(a.lw + off(k, jj, ii)) : 0.f;
    };
    // c * l(X) * factor, with the factor's loads skipped when l(X) is absent
#define PW_ADD(acc, cexpr, lam, fexpr)         \
    do {                                       \
    const float l_ = (lam);                \
    if (l_ != 0.f) acc += (cexpr) * l_ * (fexpr); \
        } while (0)
    const int k = K, j = J, i = I;
    ru = rv = rw = 0.f;

    // ---- gu: u(C) enters su (as a, b, d), sv (as b, d), sw (as b, d)
    PW_ADD(ru, tcx, LU(k, j, i + 1, nz), U(k, j, i + 1) + 2.f * U(k, j, i));
    PW_ADD(ru, tcx, LU(k, j, i, nz), U(k, j, i - 1));
    PW_ADD(ru, -tcx, LU(k, j, i - 1, nz), U(k, j, i - 1) + 2.f * U(k, j, i));
    PW_ADD(ru, -tcx, LU(k, j, i, nz), U(k, j, i + 1));
    PW_ADD(ru, tcy, LU(k, j + 1, i, nz), V(k, j, i) + V(k, j, i + 1));
    PW_ADD(ru, -tcy, LU(k, j - 1, i, nz), V(k, j - 1, i) + V(k, j - 1, i + 1));
    if (k + 1 <= nz) PW_ADD(ru, tzc1[k + 1], LU(k + 1, j, i, nz), W(k, j, i) + W(k, j, i + 1));
    if (k - 1 >= 2) PW_ADD(ru, -tzc2[k - 1], LU(k - 1, j, i, nz - 1), W(k - 1, j, i) + W(k - 1, j, i + 1));
    PW_ADD(ru, tcx, LV(k, j, i + 1, nz), V(k, j, i));
    PW_ADD(ru, tcx, LV(k, j - 1, i + 1, nz), V(k, j - 1, i));
    PW_ADD(ru, -tcx, LV(k, j, i, nz), V(k, j, i + 1));
    PW_ADD(ru, -tcx, LV(k, j - 1, i, nz), V(k, j - 1, i + 1));
    PW_ADD(ru, tcx, LW(k, j, i + 1), W(k, j, i));
    if (k - 1 >= 1) PW_ADD(ru, tcx, LW(k - 1, j, i + 1), W(k - 1, j, i));
    PW_ADD(ru, -tcx, LW(k, j, i), W(k, j, i + 1));
    if (k - 1 >= 1) PW_ADD(ru, -tcx, LW(k - 1, j, i), W(k - 1, j, i + 1));

    // ---- gv: v(C) enters su (as b, d), sv (as a, b, d), sw (as b, d)
    PW_ADD(rv, tcy, LU(k, j + 1, i, nz), U(k, j, i));
    PW_ADD(rv, tcy, LU(k, j + 1, i - 1, nz), U(k, j, i - 1));
    PW_ADD(rv, -tcy, LU(k, j, i, nz), U(k, j + 1, i));
    PW_ADD(rv, -tcy, LU(k, j, i - 1, nz), U(k, j + 1, i - 1));
    PW_ADD(rv, tcx, LV(k, j, i + 1, nz), U(k, j, i) + U(k, j + 1, i));
    PW_ADD(rv, -tcx, LV(k, j, i - 1, nz), U(k, j, i - 1) + U(k, j + 1, i - 1));
    PW_ADD(rv, tcy, LV(k, j + 1, i, nz), V(k, j + 1, i) + 2.f * V(k, j, i));
    PW_ADD(rv, tcy, LV(k, j, i, nz), V(k, j - 1, i));
    PW_ADD(rv, -tcy, LV(k, j - 1, i, nz), V(k, j - 1, i) + 2.f * V(k, j, i));
    PW_ADD(rv, -tcy, LV(k, j, i, nz), V(k, j + 1, i));
    if (k + 1 <= nz) PW_ADD(rv, tzc1[k + 1], LV(k + 1, j, i, nz), W(k, j, i) + W(k, j + 1, i));
    if (k - 1 >= 2) PW_ADD(rv, -tzc2[k - 1], LV(k - 1, j, i, nz - 1), W(k - 1, j, i) + W(k - 1, j + 1, i));
    PW_ADD(rv, tcy, LW(k, j + 1, i), W(k, j, i));
    if (k - 1 >= 1) PW_ADD(rv, tcy, LW(k - 1, j + 1, i), W(k - 1, j, i));
    PW_ADD(rv, -tcy, LW(k, j, i), W(k, j + 1, i));
    if (k - 1 >= 1) PW_ADD(rv, -tcy, LW(k - 1, j, i), W(k - 1, j + 1, i));

    // ---- gw: w(C) enters su (as b, d), sv (as b, d), sw (as a, b, d)
    if (k + 1 <= nz) {
        PW_ADD(rw, tzc1[k + 1], LU(k + 1, j, i, nz), U(k, j, i));
        PW_ADD(rw, tzc1[k + 1], LU(k + 1, j, i - 1, nz), U(k, j, i - 1));
        PW_ADD(rw, tzc1[k + 1], LV(k + 1, j, i, nz), V(k, j, i));
        PW_ADD(rw, tzc1[k + 1], LV(k + 1, j - 1, i, nz), V(k, j - 1, i));
        PW_ADD(rw, -tzc2[k], LU(k, j, i, nz - 1), U(k + 1, j, i));
        PW_ADD(rw, -tzc2[k], LU(k, j, i - 1, nz - 1), U(k + 1, j, i - 1));
        PW_ADD(rw, -tzc2[k], LV(k, j, i, nz - 1), V(k + 1, j, i));
        PW_ADD(rw, -tzc2[k], LV(k, j - 1, i, nz - 1), V(k + 1, j - 1, i));
        PW_ADD(rw, tcx, LW(k, j, i + 1), U(k, j, i) + U(k + 1, j, i));
        PW_ADD(rw, -tcx, LW(k, j, i - 1), U(k, j, i - 1) + U(k + 1, j, i - 1));
        PW_ADD(rw, tcy, LW(k, j + 1, i), V(k, j, i) + V(k + 1, j, i));
        PW_ADD(rw, -tcy, LW(k, j - 1, i), V(k, j - 1, i) + V(k + 1, j - 1, i));
        PW_ADD(rw, tzd1[k + 1], LW(k + 1, j, i), W(k + 1, j, i) + 2.f * W(k, j, i));
        PW_ADD(rw, -tzd2[k], LW(k, j, i), W(k + 1, j, i));
    }
    PW_ADD(rw, tzd1[k], LW(k, j, i), W(k - 1, j, i));
    if (k - 1 >= 2) PW_ADD(rw, -tzd2[k - 1], LW(k - 1, j, i), W(k - 1, j, i) + 2.f * W(k, j, i));
#undef PW_ADD
}

// One thread per cell: every cell the mode writes, or (RING) the interior cells
// of the first and last row and column only (nx, ny >= 3).  64 registers, so
// that four CTAs share an SM (76 registers: 273 -> 341 us at 170 x 421 x 37).
template <bool RING>
__global__ void __launch_bounds__(256, 4) adjoint_gather_kernel(const GridDev g, const AdjArgs a, const CoefDev cf) {
    const int h = a.periodic ? 0 : 1;   // extra ring of cells covered in full-array mode
    const long long wx = g.nx + 2 * h, wy = g.ny + 2 * h;
    const long long per_level = RING ? 2LL * (g.nx + g.ny - 2) : wx * wy;
    const long long total = per_level * g.nz;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        int I, J;
        const int K = 1 + (int)(idx / per_level);
        if (RING) {
            const int t = (int)(idx % per_level);
            if (t < 2 * g.nx) {
                I = 1 + t % g.nx;
                J = t < g.nx ? 1 : g.ny;
            } else {
                I = (t & 1) ? g.nx : 1;
                J = 2 + ((t - 2 * g.nx) >> 1);
            }
        } else {
            I = (int)(idx % wx) + 1 - h;
            J = (int)((idx / wx) % wy) + 1 - h;
        }
        float ru, rv, rw;
        adjoint_gather_cell(g, a, cf, K, J, I, ru, rv, rw);
        const long long c = g.origin + (long long)K * g.pk + (long long)J * g.pj + I;
        float bu = 0.f, bv = 0.f, bw = 0.f;
        if (a.accumulate) {
            bu = a.gu[c];
            bv = a.gv[c];
            bw = a.gw[c];
        } else if (a.add_lambda) {
            bu = a.lu[c];
            bv = a.lv[c];
            bw = a.lw[c];
        }
        a.gu[c] = fmaf(a.alpha, ru, bu);
        a.gv[c] = fmaf(a.alpha, rv, bv);
        a.gw[c] = fmaf(a.alpha, rw, bw);
    }
}

// ---------------------------------------------------------------------------
// TMA k-march adjoint (FP32).  A CTA owns NA*LX columns x TY rows and marches
// up the levels; one thread issues 3D TMA copies of the u, v, w and lsu, lsv,
// lsw planes (tile plus one cell all round) into a ring of S slots, each slot
// completing on its own mbarrier.  Levels K and K+1 are resident, the rest in
// flight.
//
// What a level reads.  Every term of J^T l that pairs output level K-1 with the
// cell's level K is a product of level K-1 values alone (or of them and the
// cell's own w): with
//     A(k) = lsw(i+1) w - lsw w(i+1),   B(k) = lsw(j+1) w - lsw w(j+1)
// of level k, sw's x terms give tcx (A(K) + A(K-1)) to gu and its y terms
// tcy (B(K) + B(K-1)) to gv, and su's and sv's upper terms
// -tzc2(K-1) lsu (w + w(i+1)) and -tzc2(K-1) lsv (w + w(j+1)) of level K-1.  They
// are formed at level K-1, where their factors are at hand, and carried in
// four values a cell (AdjRegs), so plane K-1 is not kept: a 3-slot ring has a
// plane in flight where the 30-row gather it replaces needed 4, and a level
// loads 16 rows of its vectors from shared memory instead of 30 (the 8 rows
// read as level K+1 are carried to be level K).
//
// What bounds it: HBM at 2048^2 x 64 (166 Gcell/s, 0.88 of 36 B a cell), below
// that the last wave and the latency of a level.  Periodic 512^2 / 1024^2 /
// 2048^2 x 64, us a call: 128 / 435 / 1616, with the 30-row gather 163 / 554 /
// 2099; open 384 x 320 x 64: 69, with the gather from global memory 978.
//
// Sensitivities count at the scheme's outputs only: interior columns (or their
// periodic images), levels 2..nz for lsu, lsv and 2..nz-1 for lsw.  Their
// tensor maps cover just those, so the copy engine's zero fill masks the rest.
//
// The full-array mode (every cell of the interior and its one-cell halo, halo
// values of u, v, w as independent inputs): tiles start at column -3 (16-byte
// aligned) and row 0, the maps of l cover the interior, the maps of u, v, w
// columns -3..nx+1 and rows 0..ny+1.  The periodic mode of a width that is no
// multiple of 4: the march writes the cells that touch no image (columns
// 2..nx-1, rows 2..ny-1; the maps of l cover the interior), and a second
// launch gathers the ring of cells around them, so the halos of l are neither
// read nor written there (511 x 512 x 64: 182 us, with the gather kernel alone 1785).
//
// CHECKED (both of these): a term whose sensitivity is exactly 0 is skipped,
// which matters where the field is not finite: a level of a thread whose result
// is not finite is not stored but redone cell by cell by adjoint_gather_cell
// after the march (any field value that is not finite makes the result so,
// zero sensitivity or not).
constexpr int kAdjPAD = 4;                       // 16-byte granule of FP32

template <int NA, int LX, int TY, int S>
struct AdjLayout {
    static_assert(NA == 2 || NA == 4, "2 or 4 cells per thread");
    static_assert(LX == 32 || LX == 16, "lanes per row");
    static constexpr int TX = LX * NA;
    static constexpr int RPW = 32 / LX;              // rows per warp
    static constexpr int WARPS = TY / RPW;
    static constexpr int THREADS = 32 * WARPS;
    static constexpr int BW = TX + 2 * kAdjPAD;
    static constexpr int ROWS = TY + 2;
    static constexpr int FIELD_RAW = BW * ROWS;
    static constexpr int FIELD = ((FIELD_RAW * 4 + 127) / 128) * 32;   // floats, 128-byte multiple
    static constexpr int STAGE = 6 * FIELD;
    static constexpr uint32_t TX_BYTES = 6u * FIELD_RAW * 4u;
    // the ring, one mbarrier per slot, 4 flag words, then the vertical
    // coefficients {tzc1, tzc2, tzd1, tzd2} of levels kb-1..ke+1 of the CTA's k
    // segment, one float4 per level (the host keeps a segment within kAdjMaxSeg
    // levels; CHECKED within kAdjMaxSegChecked)
    static constexpr size_t CTZ_OFF = (((size_t)S * STAGE * 4 + S * sizeof(uint64_t) + 16 + 15) / 16) * 16;
    static constexpr size_t SMEM = CTZ_OFF + (size_t)(kAdjMaxSeg + 2) * sizeof(float4);
};

struct AdjMaps {
    CUtensorMap m[6];   // u, v, w, lsu, lsv, lsw
};

// NA consecutive floats at a 4*NA-byte aligned address
template <int NA>
__device__ __forceinline__ void adj_ldv(const float* p, float (&o)[NA]) {
    if constexpr (NA == 4) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        o[0] = t.x;
        o[1] = t.y;
        o[2] = t.z;
        o[3] = t.w;
    } else {
        const float2 t = *reinterpret_cast<const float2*>(p);
        o[0] = t.x;
        o[1] = t.y;
    }
}
template <int NA>
__device__ __forceinline__ void adj_stv(float* p, const float (&v)[NA]) {
    if constexpr (NA == 4)
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else
        *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
}

// What a thread carries from level K to K+1: its rows of level K+1 (read at
// level K), the level-K products that enter gu and gv of level K+1, and w and
// tzd2 lsw of level K.
template <int NA>
struct AdjRegs {
    float lu[NA], lv[NA], lvm[NA], lw[NA], u[NA], v[NA], vm[NA], w[NA];   // level K; m: row j-1
    float su[NA], sv[NA], wp[NA], ep[NA];                                 // from level K-1
};

// CTAs per SM a shape's register budget is sized for: what shared memory
// allows, at most what leaves a thread 128 (4 cells) or 96 (2 cells) registers.
#ifndef PW_ADJ_REGS
#define PW_ADJ_REGS 128
#endif
template <int NA, int LX, int TY, int S>
constexpr int adj_min_blocks() {
    using L = AdjLayout<NA, LX, TY, S>;
    constexpr int by_smem = (int)((227u * 1024u) / (L::SMEM + 1024));
    constexpr int cap = 65536 / (L::THREADS * (NA == 4 ? PW_ADJ_REGS : 96));
    constexpr int m = by_smem < cap ? by_smem : cap;
    return m < 1 ? 1 : m;
}

template <int NA, int LX, int TY, int S, bool CHECKED>
__global__ void __launch_bounds__((AdjLayout<NA, LX, TY, S>::THREADS), (adj_min_blocks<NA, LX, TY, S>()))
    adjoint_march_kernel(const __grid_constant__ AdjMaps maps, const AdjArgs a, const GridDev g, const AdjGeom ge,
                         const int nseg, const CoefDev cf, int* __restrict__ err) {
    using L = AdjLayout<NA, LX, TY, S>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float* const stages = reinterpret_cast<float*>(smem_raw);
    uint64_t* const bars = reinterpret_cast<uint64_t*>(smem_raw + (size_t)S * L::STAGE * 4);
    volatile int* const abort_flag = reinterpret_cast<volatile int*>(bars + S);
    float4* const ctz = reinterpret_cast<float4*>(smem_raw + L::CTZ_OFF);   // entry k - (kb-1): level k

    const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
    const int xl = lane % LX, ty = warp * L::RPW + lane / LX;
    const int nz = g.nz, nzp2 = nz + 2;
    const int kb = 1 + (int)(((long long)blockIdx.z * nz) / nseg);
    const int ke = (int)(((long long)(blockIdx.z + 1) * nz) / nseg);
    if (ke < kb) return;
    const int pb = max(kb - 1, 1), pe = min(ke + 1, nz), np = pe - pb + 1;
    const int i_tile = (CHECKED ? ge.i0 : 1) + L::TX * blockIdx.x;   // first column and row of the tile
    const int j_tile = (CHECKED ? ge.j0 : 1) + TY * blockIdx.y;

    auto issue = [&](int p) {
        const int s = p % S, k = pb + p;
        float* dst = stages + s * L::STAGE;
        mbar_arrive_expect_tx(&bars[s], L::TX_BYTES);
#pragma unroll
        for (int f = 0; f < 3; ++f)
            tma_load_3d(dst + f * L::FIELD, &maps.m[f], i_tile - kAdjPAD + ge.fx, j_tile - 1 + ge.fy, k + ge.fz,
                        &bars[s]);
#pragma unroll
        for (int f = 3; f < 6; ++f)
            tma_load_3d(dst + f * L::FIELD, &maps.m[f], i_tile - kAdjPAD + ge.lx, j_tile - 1 + ge.ly, k + ge.lz,
                        &bars[s]);
    };
    // the issuing thread starts the first planes itself; the other warps fill
    // the table meanwhile, entries the scheme does not use as 0
    int issued = 0;
    if (tid == 0) {
        for (int s = 0; s < S; ++s) mbar_init(&bars[s], 1);
        abort_flag[0] = 0;
        fence_mbar_init();
        for (int f = 0; f < 6; ++f) prefetch_tensormap(&maps.m[f]);
        for (; issued < S && issued < np; ++issued) issue(issued);
    }
    if (tid >= 32) {
        for (int e = tid - 32; e <= ke - kb + 2; e += L::THREADS - 32) {
            const int k = kb - 1 + e;
            const bool low = k >= 2 && k <= nz, mid = k >= 2 && k < nz;
            ctz[e] = make_float4(low ? __ldg(cf.tz + k) : 0.f, mid ? __ldg(cf.tz + nzp2 + k) : 0.f,
                                 mid ? __ldg(cf.tz + 2 * nzp2 + k) : 0.f, mid ? __ldg(cf.tz + 3 * nzp2 + k) : 0.f);
        }
    }
    __syncthreads();

    const float tcx = cf.tcx, tcy = cf.tcy;
    const int J = j_tile + ty, I0 = i_tile + NA * xl;
    const int c0 = (ty + 1) * L::BW + kAdjPAD + NA * xl;   // the thread's vector in a staged field
    const int ilo = CHECKED ? ge.ilo : 1, ihi = CHECKED ? ge.ihi : g.nx;
    const bool valid = (!CHECKED || (J >= ge.jlo && I0 + NA > ilo)) && J <= (CHECKED ? ge.jhi : g.ny) && I0 <= ihi;
    const bool whole = I0 >= ilo && I0 + NA - 1 <= ihi;
    // sensitivities as the caller gave them: staged where they count, else in memory
    const bool staged = !CHECKED || (J >= 1 && J <= g.ny && I0 >= 1 && I0 + NA - 1 <= g.nx);
    const bool left = CHECKED && I0 < 0;   // columns -3..-1 hold padding
    const long long row_off = g.origin + (long long)J * g.pj + I0;
    const unsigned FULL = 0xffffffffu;
    int waited = 0;
    unsigned long long redo = 0;   // CHECKED: levels kb + bit whose result was not finite

    AdjRegs<NA> st;
#pragma unroll
    for (int c = 0; c < NA; ++c) st.su[c] = st.sv[c] = st.wp[c] = st.ep[c] = 0.f;

    enum { U = 0, V = 1, W = 2, LU = 3, LV = 4, LW = 5 };
    // One level; returns false on abort.  FAST: 3 <= K <= nz-2 and K > pb, where every term exists.
    auto level = [&](const int K, auto fast) -> bool {
        constexpr bool FAST = decltype(fast)::value;
        const int lp = K - pb;
        const bool up = FAST || K + 1 <= nz;
        bool ok = true;
        if (!FAST && lp == 0) ok = mbar_wait_bounded(&bars[0], 0, kWaitLimitNs);
        if (ok && up) ok = mbar_wait_bounded(&bars[(lp + 1) % S], (uint32_t)(((lp + 1) / S) & 1), kWaitLimitNs);
        ok = __all_sync(FULL, ok);
        if (!ok) abort_flag[0] = 1;
        if (ok) {
            waited = lp + (up ? 2 : 1);
            const float* const P0 = stages + (lp % S) * L::STAGE + c0;         // level K
            const float* const P1 = stages + ((lp + 1) % S) * L::STAGE + c0;   // level K+1
            auto row = [&](const float* P, int f, int dj, float (&x)[NA]) {
                adj_ldv<NA>(P + f * L::FIELD + dj * L::BW, x);
                if (left && f < LU) {
#pragma unroll
                    for (int c = 0; c < NA; ++c)
                        if (I0 + c < 0) x[c] = 0.f;
                }
            };
            // the value left (m) and right (p) of the thread's vector: from the
            // neighbouring lane, at the row's ends from the staged row (every
            // lane loading it: 1652 -> 1759 us at 2048^2 x 64)
            auto nm = [&](const float* P, int f, int dj, const float (&x)[NA]) {
                float t = __shfl_up_sync(FULL, x[NA - 1], 1, LX);
                if (xl == 0) t = P[f * L::FIELD + dj * L::BW - 1];
                return t;
            };
            auto np_ = [&](const float* P, int f, int dj, const float (&x)[NA]) {
                float t = __shfl_down_sync(FULL, x[0], 1, LX);
                if (xl == LX - 1) t = P[f * L::FIELD + dj * L::BW + NA];
                return t;
            };
            auto at = [](const float (&x)[NA], float m, float p, int c) { return c < 0 ? m : (c < NA ? x[c] : p); };
            if (!FAST && lp == 0) {
                row(P0, LU, 0, st.lu);
                row(P0, LV, 0, st.lv);
                row(P0, LV, -1, st.lvm);
                row(P0, LW, 0, st.lw);
                row(P0, U, 0, st.u);
                row(P0, V, 0, st.v);
                row(P0, V, -1, st.vm);
                row(P0, W, 0, st.w);
            }
            const float4 z0 = ctz[K - kb + 1], z1 = ctz[K - kb + 2];   // levels K, K+1
            // products of level K that enter this level and the next
            float A[NA], B[NA], PX[NA], PY[NA], wq[NA], lwq[NA];
            const float wr = np_(P0, W, 0, st.w), lwr = np_(P0, LW, 0, st.lw);
            row(P0, W, 1, wq);
            row(P0, LW, 1, lwq);
#pragma unroll
            for (int c = 0; c < NA; ++c) {
                const float wn = at(st.w, 0.f, wr, c + 1), lwn = at(st.lw, 0.f, lwr, c + 1);
                PX[c] = st.w[c] + wn;
                PY[c] = st.w[c] + wq[c];
                A[c] = fmaf(lwn, st.w[c], -st.lw[c] * wn);
                B[c] = fmaf(lwq[c], st.w[c], -st.lw[c] * wq[c]);
            }
            // level K+1 rows (carried)
            AdjRegs<NA> nx;
            if (up) {
                row(P1, LU, 0, nx.lu);
                row(P1, LV, 0, nx.lv);
            } else {
#pragma unroll
                for (int c = 0; c < NA; ++c)
                    nx.lu[c] = nx.lv[c] = nx.lvm[c] = nx.lw[c] = nx.u[c] = nx.v[c] = nx.vm[c] = nx.w[c] = 0.f;
            }
            if (FAST || K >= kb) {
                const float c1p = z1.x, c2 = z0.y, d1p = z1.z, d1 = z0.z, d2 = z0.w;
                const long long o = row_off + (long long)K * g.pk;
                float base[NA], r0[NA], r1[NA], r2[NA];
                // one field's result: g = alpha r + base
                auto finish = [&](float* __restrict__ gp, const float* __restrict__ lp_, const float (&l)[NA],
                                  float (&r)[NA]) {
                    if (a.accumulate || (a.add_lambda && !(staged && (FAST || (K >= 2 && K < nz))))) {
                        const float* q = (a.accumulate ? gp : lp_) + o;
                        if (valid && whole) {
                            adj_ldv<NA>(q, base);
                        } else {
#pragma unroll
                            for (int c = 0; c < NA; ++c)
                                base[c] = (valid && I0 + c >= ilo && I0 + c <= ihi) ? q[c] : 0.f;
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < NA; ++c) base[c] = a.add_lambda ? l[c] : 0.f;
                    }
#pragma unroll
                    for (int c = 0; c < NA; ++c) r[c] = fmaf(a.alpha, r[c], base[c]);
                };
                auto store = [&](float* __restrict__ gp, const float (&r)[NA]) {
                    if (!valid) return;
                    if (whole) {
                        adj_stv<NA>(gp + o, r);
                    } else {
#pragma unroll
                        for (int c = 0; c < NA; ++c)
                            if (I0 + c >= ilo && I0 + c <= ihi) gp[o + c] = r[c];
                    }
                };
                // ---- gu: u in su (as a, b, d), in sv and sw (as b, d)
                const float ul = nm(P0, U, 0, st.u), ur = np_(P0, U, 0, st.u);
                const float lul = nm(P0, LU, 0, st.lu), lur = np_(P0, LU, 0, st.lu);
                const float vr = np_(P0, V, 0, st.v), lvr = np_(P0, LV, 0, st.lv);
                const float vmr = np_(P0, V, -1, st.vm), lvmr = np_(P0, LV, -1, st.lvm);
                float luq[NA], lum[NA];
                row(P0, LU, 1, luq);
                row(P0, LU, -1, lum);
#pragma unroll
                for (int c = 0; c < NA; ++c) {
                    const float um = at(st.u, ul, ur, c - 1), up_ = at(st.u, ul, ur, c + 1);
                    const float vn = at(st.v, 0.f, vr, c + 1), vmn = at(st.vm, 0.f, vmr, c + 1);
                    float x = at(st.lu, lul, lur, c + 1) * fmaf(2.f, st.u[c], up_);
                    x = fmaf(-at(st.lu, lul, lur, c - 1), fmaf(2.f, st.u[c], um), x);
                    x = fmaf(st.lu[c], um - up_, x);
                    x = fmaf(at(st.lv, 0.f, lvr, c + 1), st.v[c], x);
                    x = fmaf(-st.lv[c], vn, x);
                    x = fmaf(at(st.lvm, 0.f, lvmr, c + 1), st.vm[c], x);
                    x = fmaf(-st.lvm[c], vmn, x);
                    x += A[c];
                    const float y = fmaf(luq[c], st.v[c] + vn, -lum[c] * (st.vm[c] + vmn));
                    r0[c] = fmaf(tcx, x, fmaf(tcy, y, st.su[c]));
                    if (up) r0[c] = fmaf(c1p * nx.lu[c], PX[c], r0[c]);
                }
                finish(a.gu, a.lu, st.lu, r0);
                if (!CHECKED) store(a.gu, r0);
                // ---- gv: v in su (as b, d), in sv (as a, b, d), in sw (as b, d)
                float uq[NA], vq[NA], lvq[NA];
                row(P0, U, 1, uq);
                row(P0, V, 1, vq);
                row(P0, LV, 1, lvq);
                const float uql = nm(P0, U, 1, uq), luql = nm(P0, LU, 1, luq), lvl = nm(P0, LV, 0, st.lv);
                // sv's y terms as seen from v; u(j) + u(j+1): cell c and its left neighbour
                float D = fmaf(luql, ul, -lul * uql), Q = ul + uql;
#pragma unroll
                for (int c = 0; c < NA; ++c) {
                    const float Dn = fmaf(luq[c], st.u[c], -st.lu[c] * uq[c]), Qn = st.u[c] + uq[c];
                    const float x = fmaf(at(st.lv, lvl, lvr, c + 1), Qn, -at(st.lv, lvl, lvr, c - 1) * Q);
                    float y = D + Dn;
                    y = fmaf(lvq[c], fmaf(2.f, st.v[c], vq[c]), y);
                    y = fmaf(-st.lvm[c], fmaf(2.f, st.v[c], st.vm[c]), y);
                    y = fmaf(st.lv[c], st.vm[c] - vq[c], y);
                    y += B[c];
                    r1[c] = fmaf(tcx, x, fmaf(tcy, y, st.sv[c]));
                    if (up) r1[c] = fmaf(c1p * nx.lv[c], PY[c], r1[c]);
                    D = Dn;
                    Q = Qn;
                }
                finish(a.gv, a.lv, st.lv, r1);
                if (!CHECKED) store(a.gv, r1);
                // ---- gw: w in su, sv (as b, d), in sw (as a, b, d)
                if (up) {
                    row(P1, U, 0, nx.u);
                    row(P1, V, 0, nx.v);
                    row(P1, V, -1, nx.vm);
                    row(P1, LV, -1, nx.lvm);
                    row(P1, W, 0, nx.w);
                    row(P1, LW, 0, nx.lw);
                }
                // terms with level K-1: the cell's own w and lsw there
#pragma unroll
                for (int c = 0; c < NA; ++c) {
                    float t = 0.f;
                    if (FAST || K >= 2) t = d1 * st.lw[c] * st.wp[c];
                    if (FAST || (K >= 3 && K <= nz)) t = fmaf(-st.ep[c], fmaf(2.f, st.w[c], st.wp[c]), t);
                    r2[c] = t;
                }
                if (up) {
                    float lwm[NA];
                    row(P0, LW, -1, lwm);
                    const float lwl = nm(P0, LW, 0, st.lw);
                    const float unl = nm(P1, U, 0, nx.u), lunl = nm(P1, LU, 0, nx.lu);
                    // su's upper terms at K+1 and K as seen from w; u(k) + u(k+1)
                    float F = lunl * ul, G = lul * unl, R = ul + unl;
#pragma unroll
                    for (int c = 0; c < NA; ++c) {
                        const float Fn = nx.lu[c] * st.u[c], Gn = st.lu[c] * nx.u[c], Rn = st.u[c] + nx.u[c];
                        float e1 = F + Fn;
                        e1 = fmaf(nx.lv[c], st.v[c], e1);
                        e1 = fmaf(nx.lvm[c], st.vm[c], e1);
                        float e2 = G + Gn;
                        e2 = fmaf(st.lv[c], nx.v[c], e2);
                        e2 = fmaf(st.lvm[c], nx.vm[c], e2);
                        const float ex = fmaf(at(st.lw, lwl, lwr, c + 1), Rn, -at(st.lw, lwl, lwr, c - 1) * R);
                        const float ey = fmaf(lwq[c], st.v[c] + nx.v[c], -lwm[c] * (st.vm[c] + nx.vm[c]));
                        float t = fmaf(tcx, ex, fmaf(tcy, ey, fmaf(-c2, e2, -d2 * st.lw[c] * nx.w[c])));
                        t = fmaf(c1p, e1, t);
                        if (FAST || K + 1 < nz) t = fmaf(d1p * nx.lw[c], fmaf(2.f, st.w[c], nx.w[c]), t);
                        r2[c] += t;
                        F = Fn;
                        G = Gn;
                        R = Rn;
                    }
                }
                finish(a.gw, a.lw, st.lw, r2);
                if (!CHECKED) {
                    store(a.gw, r2);
                } else {
                    float t = 0.f;   // stays 0 while every result is finite
#pragma unroll
                    for (int c = 0; c < NA; ++c)
                        if (I0 + c >= ilo && I0 + c <= ihi) t = fmaf(r0[c], 0.f, fmaf(r1[c], 0.f, fmaf(r2[c], 0.f, t)));
                    if (t == 0.f) {
                        store(a.gu, r0);
                        store(a.gv, r1);
                        store(a.gw, r2);
                    } else if (valid) {
                        redo |= 1ull << (K - kb);
                    }
                }
            } else if (up) {   // a segment's priming level: the rows of its first level
                row(P1, U, 0, nx.u);
                row(P1, V, 0, nx.v);
                row(P1, V, -1, nx.vm);
                row(P1, LV, -1, nx.lvm);
                row(P1, W, 0, nx.w);
                row(P1, LW, 0, nx.lw);
            }
            // roll to level K+1
            const float c2n = z0.y, d2n = z0.w;
#pragma unroll
            for (int c = 0; c < NA; ++c) {
                const bool mid = FAST || (K >= 2 && K < nz);
                nx.su[c] = mid ? fmaf(tcx, A[c], -c2n * st.lu[c] * PX[c]) : 0.f;
                nx.sv[c] = mid ? fmaf(tcy, B[c], -c2n * st.lv[c] * PY[c]) : 0.f;
                nx.wp[c] = st.w[c];
                nx.ep[c] = d2n * st.lw[c];
            }
            st = nx;
        }
        __syncthreads();
        if (abort_flag[0]) return false;
        if (tid == 0 && issued < np && issued <= lp + S) {   // plane K is free
            fence_proxy_async_smem();
            issue(issued);
            ++issued;
        }
        return true;
    };

    using Fast = std::integral_constant<bool, true>;
    using Gen = std::integral_constant<bool, false>;
    bool aborted = false;
    int K = pb;
    for (; K <= ke && (K == pb || K < 3) && !aborted; ++K) aborted = !level(K, Gen{});
    constexpr int kUnroll = CHECKED ? 2 : 1;   // (2: open 69.3 -> 67.9 us at 384 x 320 x 64, periodic 1616 -> 1627 at 2048^2)
#pragma unroll kUnroll
    for (; K <= min(ke, nz - 2) && !aborted; ++K) aborted = !level(K, Fast{});
    for (; K <= ke && !aborted; ++K) aborted = !level(K, Gen{});
    if (aborted && tid == 0) {
        report_error(err, DEV_TIMEOUT_TMA_WAIT);
        // let the copies still in flight land before the CTA's smem is released
        for (int p = waited; p < issued; ++p)
            if (!mbar_wait_bounded(&bars[p % S], (uint32_t)((p / S) & 1), kDrainLimitNs)) break;
    }
    if constexpr (CHECKED) {
        while (redo && !aborted) {
            const int Kr = kb + __ffsll((long long)redo) - 1;
            redo &= redo - 1;
            for (int I = max(I0, ilo); I <= min(I0 + NA - 1, ihi); ++I) {
                float r[3];
                adjoint_gather_cell(g, a, cf, Kr, J, I, r[0], r[1], r[2]);
                const long long o = row_off + (long long)Kr * g.pk + (I - I0);
                a.gu[o] = fmaf(a.alpha, r[0], a.accumulate ? a.gu[o] : (a.add_lambda ? a.lu[o] : 0.f));
                a.gv[o] = fmaf(a.alpha, r[1], a.accumulate ? a.gv[o] : (a.add_lambda ? a.lv[o] : 0.f));
                a.gw[o] = fmaf(a.alpha, r[2], a.accumulate ? a.gw[o] : (a.add_lambda ? a.lw[o] : 0.f));
            }
        }
    }
}

// Launch shapes: the ones pw_set_adjoint_config takes (32 lanes per row,
// periodic mode), and the automatic one (cells, lanes, rows, slots): four CTAs
// of 4 warps per SM.  Periodic 512^2 / 1024^2 / 2048^2 x 64 and open 384 x 320 x 64:
// 128 / 435 / 1616 / 69 us, 32 lanes x 8 rows (two CTAs of 8 warps) 129 / 445 / 1652 /
// 85, 16 x 16 130 / 449 / 1678 / 71; at 168 registers 32 x 8 takes 154 / 539 / 2051 / 78.
#define PW_ADJ_CONFIGS(X) X(4, 5, 4) X(4, 4, 4) X(4, 6, 4) X(2, 4, 4) X(2, 5, 4) X(2, 6, 4) X(2, 8, 4) X(2, 8, 3)
#define PW_ADJ_AUTO(X) X(4, 16, 8, 3)

AdjConfig adjoint_shape(const AdjConfig& u) {
    AdjConfig c{u.na ? u.na : 4, u.ty ? u.ty : 6, u.stages ? u.stages : 4, u.nseg, 32};
    if (c.na == 4 && c.ty == 8 && c.stages == 3) c.lx = 16;
    return c;
}

bool adjoint_config_supported(const AdjConfig& c) {
#define PW_AB(NA_, LX_, TY_, S_) \
    if (c.lx == LX_ && c.na == NA_ && c.ty == TY_ && c.stages == S_) return true;
    PW_ADJ_AUTO(PW_AB)
#undef PW_AB
#define PW_AS(NA_, TY_, S_) \
    if (c.lx == 32 && c.na == NA_ && c.ty == TY_ && c.stages == S_) return true;
    PW_ADJ_CONFIGS(PW_AS)
#undef PW_AS
    return false;
}

template <int NA, int LX, int TY, int S, bool CHECKED>
static cudaError_t adj_inst(const AdjConfig& c, int* bps, const GridDev& g, const AdjGeom& ge, const AdjMaps& m,
                            const AdjArgs& a, const CoefDev& cf, int* err, cudaStream_t s) {
    using L = AdjLayout<NA, LX, TY, S>;
    auto kern = adjoint_march_kernel<NA, LX, TY, S, CHECKED>;
    cudaError_t e = set_smem_attr_once(kern, (int)L::SMEM);
    if (e != cudaSuccess) return e;
    if (bps) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, kern, L::THREADS, L::SMEM);
    constexpr int most = CHECKED ? kAdjMaxSegChecked : kAdjMaxSeg;
    const int nseg = std::max(c.nseg, (g.nz + most - 1) / most);
    const int wx = ge.ihi - ge.i0 + 1, wy = ge.jhi - ge.j0 + 1;
    dim3 grid((wx + L::TX - 1) / L::TX, (wy + TY - 1) / TY, nseg);
    kern<<<grid, dim3(32, L::WARPS), L::SMEM, s>>>(m, a, g, ge, nseg, cf, err);
    return cudaGetLastError();
}

static cudaError_t adj_dispatch(const AdjConfig& c, bool checked, int* bps, const GridDev& g, const AdjGeom& ge,
                                const AdjMaps& m, const AdjArgs& a, const CoefDev& cf, int* err, cudaStream_t s) {
#define PW_AA(NA_, LX_, TY_, S_)                                                                      \
    if (c.na == NA_ && c.lx == LX_ && c.ty == TY_ && c.stages == S_)                                  \
        return checked ? adj_inst<NA_, LX_, TY_, S_, true>(c, bps, g, ge, m, a, cf, err, s)              \
                    : adj_inst<NA_, LX_, TY_, S_, false>(c, bps, g, ge, m, a, cf, err, s);
    PW_ADJ_AUTO(PW_AA)
#undef PW_AA
#define PW_AD(NA_, TY_, S_)                                                                           \
    if (!checked && c.lx == 32 && c.na == NA_ && c.ty == TY_ && c.stages == S_)                          \
        return adj_inst<NA_, 32, TY_, S_, false>(c, bps, g, ge, m, a, cf, err, s);
    PW_ADJ_CONFIGS(PW_AD)
#undef PW_AD
    return cudaErrorInvalidConfiguration;
}

int adjoint_blocks_per_sm(const AdjConfig& c, bool checked) {
    int n = 0;
    if (adj_dispatch(c, checked, &n, GridDev{}, AdjGeom{}, AdjMaps{}, AdjArgs{}, CoefDev{}, nullptr, nullptr) != cudaSuccess)
        return 0;
    return n;
}

cudaError_t launch_adjoint_tma(const GridDev& g, const AdjGeom& ge, AdjMode mode, const CUtensorMap* maps6,
                               const float* const* q6, float* const* g3, float alpha, int accumulate, int add_lambda,
                               const CoefDev& cf, int* err, const AdjConfig& c, int num_sms, cudaStream_t s) {
    AdjMaps m;
    for (int f = 0; f < 6; ++f) m.m[f] = maps6[f];
    const AdjArgs a{q6[0], q6[1], q6[2], q6[3], q6[4], q6[5], g3[0], g3[1], g3[2], alpha, accumulate, add_lambda,
                    mode != ADJ_OPEN};
    cudaError_t e = adj_dispatch(c, mode != ADJ_PERIODIC, nullptr, g, ge, m, a, cf, err, s);
    if (e == cudaSuccess && mode == ADJ_PERIODIC_ANY) {
        const long long ring = 2LL * (g.nx + g.ny - 2) * g.nz;
        adjoint_gather_kernel<true><<<(unsigned)std::min<long long>((ring + 255) / 256, num_sms * 16), 256, 0, s>>>(g, a, cf);
        e = cudaGetLastError();
    }
    return e;
}

cudaError_t launch_adjoint(const GridDev& g, const float* u, const float* v, const float* w, const float* lu,
                           const float* lv, const float* lw, float* gu, float* gv, float* gw, float alpha,
                           int accumulate, int add_lambda, int periodic, const CoefDev& cf, int num_sms,
                           cudaStream_t s) {
    AdjArgs a{u, v, w, lu, lv, lw, gu, gv, gw, alpha, accumulate, add_lambda, periodic};
    const int hh = periodic ? 0 : 1;
    const long long total = (long long)(g.nx + 2 * hh) * (g.ny + 2 * hh) * g.nz;
    const int threads = 256;
    long long blocks = (total + threads - 1) / threads;
    if (blocks > (long long)num_sms * 16) blocks = (long long)num_sms * 16;
    if (blocks < 1) blocks = 1;
    adjoint_gather_kernel<false><<<(unsigned)blocks, threads, 0, s>>>(g, a, cf);
    return cudaGetLastError();
}

}  // namespace pw
