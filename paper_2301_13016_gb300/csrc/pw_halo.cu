// Periodic lateral halo swap of one field (the doubly periodic boundary the
// scheme needs before each evaluation, Sec. 2.2).
#include <algorithm>

#include "pw_device.cuh"
#include "pw_internal.h"

namespace pw {

// One thread per halo cell of levels 1..nz.  Every halo cell copies its
// periodic image directly (i' = 1 + (i-1) mod nx, likewise j), which equals
// the x-then-y two-pass swap including the corners.  Pure element copies in
// the storage type (E = 4 or 2 bytes).
// blockIdx.y = field: one launch for the fields of a state (three fields at
// 512^2 x 64: 9.9 us in three launches, 5.9 in one).
struct HaloFields {
    void* f[3];
};
template <typename E>
__global__ void fill_halo_kernel(const GridDev g, const HaloFields fs) {
    E* __restrict__ const f = reinterpret_cast<E*>(fs.f[blockIdx.y]);
    const int h = g.halo;
    const long long wx = g.nx + 2 * h;
    const long long rows = 2LL * h * wx;              // halo rows, full width
    const long long cols = 2LL * h * g.ny;            // halo columns of interior rows
    const long long per_level = rows + cols;
    const long long total = per_level * g.nz;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int k = 1 + (int)(idx / per_level);
        long long t = idx % per_level;
        int i, j;
        if (t < rows) {
            const int b = (int)(t / wx);
            i = 1 - h + (int)(t % wx);
            j = (b < h) ? (1 - h + b) : (g.ny + 1 + b - h);
        } else {
            t -= rows;
            const int b = (int)(t / g.ny);
            j = 1 + (int)(t % g.ny);
            i = (b < h) ? (1 - h + b) : (g.nx + 1 + b - h);
        }
        const int si = 1 + (((i - 1) % g.nx) + g.nx) % g.nx;
        const int sj = 1 + (((j - 1) % g.ny) + g.ny) % g.ny;
        const long long base = g.origin + (long long)k * g.pk;
        f[base + (long long)j * g.pj + i] = f[base + (long long)sj * g.pj + si];
    }
}

cudaError_t launch_fill_halo(pw_dtype_t dt, const GridDev& g, void* const* f, int n, int num_sms, cudaStream_t s) {
    const long long per_level = 2LL * g.halo * (g.nx + 2 * g.halo) + 2LL * g.halo * g.ny;
    const long long total = per_level * g.nz;
    const int threads = 256;
    long long blocks = (total + threads - 1) / threads;
    if (blocks > (long long)num_sms * 8) blocks = (long long)num_sms * 8;
    if (blocks < 1) blocks = 1;
    HaloFields fs{};
    for (int q = 0; q < n; ++q) fs.f[q] = f[q];
    const dim3 grid((unsigned)blocks, (unsigned)n);
    if (dtype_size(dt) == 4)
        fill_halo_kernel<uint32_t><<<grid, threads, 0, s>>>(g, fs);
    else
        fill_halo_kernel<uint16_t><<<grid, threads, 0, s>>>(g, fs);
    return cudaGetLastError();
}

// dst = src on the interior of levels 1..nz, 0 in every other of the first n
// elements (halos, z halos, padding); src 0: zeros; dst may be src.  blockIdx.y
// = field; a warp takes one padded row after another (from its column i = 0 to
// the next row's, the first from element 0, the last to element n), so the only
// division is one per row, and copies its interior 16 bytes a lane where the
// buffers and rows are aligned (V > 1).  HBM-bound:
// three fields at 512^2 x 64 76 us, in place 34, where torch's mask and selects
// took 191, a mask and masked fills 135; one thread per element, two divisions
// each, took 182 and 147.
struct KeepFields {
    const void* src[3];
    void* dst[3];
};
template <typename E, int V>
struct alignas(sizeof(E) * V) KeepVec {
    E x[V];
};
template <typename E, int V>
__global__ void keep_interior_kernel(const GridDev g, const KeepFields fs, const long long n) {
    const E* const src = reinterpret_cast<const E*>(fs.src[blockIdx.y]);
    E* const dst = reinterpret_cast<E*>(fs.dst[blockIdx.y]);
    const bool in_place = static_cast<const void*>(src) == static_cast<const void*>(dst);
    using Vec = KeepVec<E, V>;
    const int lane = threadIdx.x & 31;
    const int rows = g.ny + 2 * g.halo, total = rows * (g.nz + 2);
    auto start = [&](int q) {   // element (k, j, i = 0) of padded row q
        const int k = q / rows;
        return g.origin + (long long)k * g.pk + (long long)(q - k * rows + 1 - g.halo) * g.pj;
    };
    for (int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < total; q += (gridDim.x * blockDim.x) >> 5) {
        const int k = q / rows, j = q - k * rows + 1 - g.halo;
        const long long s0 = start(q), lo = q ? s0 : 0, hi = q + 1 < total ? start(q + 1) : n;
        const bool inner = k >= 1 && k <= g.nz && j >= 1 && j <= g.ny;
        const long long a = inner ? s0 + 1 : hi, b = inner ? s0 + 1 + g.nx : hi;   // the interior: [a, b)
        auto zero = [&](long long x, const long long y) {
            if constexpr (V > 1) {   // single elements up to a vector's boundary, then whole vectors
                const long long x1 = min(y, (x + V - 1) / V * V);
                for (long long e = x + lane; e < x1; e += 32) dst[e] = E(0);
                Vec t;
#pragma unroll
                for (int c = 0; c < V; ++c) t.x[c] = E(0);
                for (long long e = x1 + lane * V; e + V <= y; e += 32 * V) *reinterpret_cast<Vec*>(dst + e) = t;
                x = x1 + (y - x1) / V * V;
            }
            for (long long e = x + lane; e < y; e += 32) dst[e] = E(0);
        };
        zero(lo, a);
        if (inner && !in_place) {
            long long e1 = a;
            if (V > 1 && a % V == 0) {
                for (long long e = a + lane * V; e + V <= b; e += 32 * V) {
                    Vec t;
                    if (src) {
                        t = *reinterpret_cast<const Vec*>(src + e);
                    } else {
#pragma unroll
                        for (int c = 0; c < V; ++c) t.x[c] = E(0);
                    }
                    *reinterpret_cast<Vec*>(dst + e) = t;
                }
                e1 = a + (b - a) / V * V;
            }
            for (long long e = e1 + lane; e < b; e += 32) dst[e] = src ? src[e] : E(0);
        }
        zero(b, hi);
    }
}

cudaError_t launch_keep_interior(pw_dtype_t dt, const GridDev& g, const void* const* src, void* const* dst, long long n,
                                 int num_sms, cudaStream_t s) {
    KeepFields fs{};
    for (int q = 0; q < 3; ++q) {
        fs.src[q] = src[q];
        fs.dst[q] = dst[q];
    }
    bool vec = true;   // every buffer on a 16-byte boundary
    for (int q = 0; q < 3; ++q)
        vec = vec && (reinterpret_cast<uintptr_t>(src[q]) & 15) == 0 && (reinterpret_cast<uintptr_t>(dst[q]) & 15) == 0;
    const int es = (int)dtype_size(dt), threads = 256;
    const long long warps = (long long)(g.ny + 2 * g.halo) * (g.nz + 2);
    const dim3 grid((unsigned)std::max(1LL, std::min<long long>((warps + 7) / 8, (long long)num_sms * 16)), 3);
    if (es == 4 && vec)
        keep_interior_kernel<uint32_t, 4><<<grid, threads, 0, s>>>(g, fs, n);
    else if (es == 4)
        keep_interior_kernel<uint32_t, 1><<<grid, threads, 0, s>>>(g, fs, n);
    else if (vec)
        keep_interior_kernel<uint16_t, 8><<<grid, threads, 0, s>>>(g, fs, n);
    else
        keep_interior_kernel<uint16_t, 1><<<grid, threads, 0, s>>>(g, fs, n);
    return cudaGetLastError();
}

}  // namespace pw
