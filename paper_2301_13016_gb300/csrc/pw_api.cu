// C ABI of the PW library: handles, argument validation, TMA descriptors,
// kernel selection and launch.  See include/pw.h for the contract.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <atomic>
#include <mutex>
#include <string>
#include <vector>

#include "pw_device.cuh"
#include "pw_internal.h"

namespace pw {

size_t dtype_size(pw_dtype_t t) { return t == PW_F32 ? 4 : 2; }

static thread_local std::string g_err;

static pw_status_t fail(pw_status_t s, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return s;
}

static pw_status_t cuda_fail(cudaError_t e, const char* what) {
    return fail(e == cudaErrorMemoryAllocation ? PW_ERR_OOM : PW_ERR_CUDA, "%s: %s (%s)", what,
                cudaGetErrorString(e), cudaGetErrorName(e));
}

#define PW_CUDA(call, what)                          \
    do {                                             \
        cudaError_t e_ = (call);                     \
        if (e_ != cudaSuccess) return cuda_fail(e_, what); \
    } while (0)

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// dependency on libcuda).
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// Which cells of a field a tensor map covers: the whole padded field (the
// k-march), or one of the adjoint's (adj_map).
enum { MAP_FIELD = 0, MAP_ADJ = 1 };
struct MapCacheEntry {
    const void* ptr = nullptr;
    int kind = MAP_FIELD;
    int box_w = 0, box_h = 0;
    CUtensorMap map;
};

}  // namespace pw

using namespace pw;

struct pw_handle_s {
    pw_grid_t grid;
    int device = 0;
    int num_sms = 0;
    float tcx = 0.f, tcy = 0.f;
    float* d_tz = nullptr;      // tzc1 | tzc2 | tzd1 | tzd2, nz+2 each
    int* d_err = nullptr;       // device status word (bounded-wait timeouts)
    int kernel_kind = 0;        // 0 auto, 1 generic, 2 TMA
    int last_kernel = 0;
    // user overrides: every field 0 = automatic (nc and rp too, whose struct
    // defaults are the values a launch uses)
    TmaConfig tma_user{0, 0, 0, 0, 0, 0, 0, 0};
    TmaConfig tma_auto[2] = {{0, 0, 0, 0}, {0, 0, 0, 0}};   // per mode (source terms, steps); ty == 0: not chosen yet
    int steps_per_pass = 0;           // pw_step temporal blocking: 0 auto (= 1), 1, 2
    Step2Config step2_user{0, 0, 0, 0};
    Step2Config step2_auto{0, 0, 0, 0};   // ty == 0: not chosen yet
    AdjConfig adj_user{0, 0, 0, 0};       // TMA adjoint shape; 0 = automatic
    AdjConfig adj_auto[3] = {};           // the shape in use, per AdjMode; na == 0: not chosen yet
    MapCacheEntry maps[8];
    int map_next = 0;   // round-robin replacement
    // field pointers already found to be device memory of this handle's GPU
    static constexpr int kDevCache = 32;
    const void* dev_ok[kDevCache] = {};
    int dev_next = 0;
    // pw_tendencies_host staging and its copy / compute pipeline
    void* d_stage[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    cudaStream_t hs[3] = {nullptr, nullptr, nullptr};   // copy in, compute, copy out
    static constexpr int kMaxChunks = 32;
    cudaEvent_t ev_in[kMaxChunks] = {}, ev_comp[kMaxChunks] = {}, ev_out[kMaxChunks] = {};
    cudaEvent_t ev_start = nullptr, ev_end = nullptr;
    bool host_prev_plain = false;   // the last host-path call took the one-launch path (it recorded ev_end on its stream)
    // validation scratch: 4*(nblocks+1) doubles + wk (nz+2 doubles)
    double* d_scratch = nullptr;
    int nblocks = 0;
};

static GridDev to_dev(const pw_grid_t& g) {
    GridDev d;
    d.nx = g.nx;
    d.ny = g.ny;
    d.nz = g.nz;
    d.halo = g.halo;
    d.pj = g.pitch_j;
    d.pk = g.pitch_k;
    d.origin = g.origin;
    return d;
}

// Element count a field allocation must hold for this layout.
static long long alloc_elems_of(const pw_grid_t& g) {
    return g.origin + (long long)(g.nz + 1) * g.pitch_k + (long long)(g.ny + g.halo) * g.pitch_j + g.nx + g.halo +
           1;
}

pw_status_t pw::validate_grid(const pw_grid_t* g) {
    if (!g) return fail(PW_ERR_ARG, "grid is NULL");
    if (g->dtype != PW_F32 && g->dtype != PW_BF16 && g->dtype != PW_F16)
        return fail(PW_ERR_ARG, "unknown dtype %d", (int)g->dtype);
    if (g->nx < 1 || g->ny < 1) return fail(PW_ERR_ARG, "nx, ny must be >= 1 (got %d, %d)", g->nx, g->ny);
    if (g->nz < 3) return fail(PW_ERR_ARG, "nz must be >= 3 (got %d)", g->nz);
    if (g->halo < 1) return fail(PW_ERR_ARG, "halo must be >= 1 (got %d)", g->halo);
    if (g->halo > g->nx || g->halo > g->ny)
        return fail(PW_ERR_ARG, "halo %d exceeds the interior (%d x %d)", g->halo, g->nx, g->ny);
    if (g->pitch_j < (long long)g->nx + 2 * g->halo)
        return fail(PW_ERR_ARG, "pitch_j %lld < nx + 2*halo", (long long)g->pitch_j);
    if (g->pitch_k < g->pitch_j * ((long long)g->ny + 2 * g->halo))
        return fail(PW_ERR_ARG, "pitch_k %lld < pitch_j*(ny + 2*halo)", (long long)g->pitch_k);
    if (g->origin < (long long)(g->halo - 1) * (g->pitch_j + 1))
        return fail(PW_ERR_ARG, "origin %lld leaves no room for the halo", (long long)g->origin);
    return PW_OK;
}

// TMA eligibility of the layout (pointer alignment is checked per call).
// Writes the x offset `ox` of element i = 0 within its padded row.
bool pw::tma_layout_ok(const pw_grid_t& g, int* ox_out, const char** why, bool any_nx) {
    const long long es = (long long)dtype_size(g.dtype);
    const long long padx = 16 / es;
    if (!any_nx && g.nx % 4) { *why = "nx is not a multiple of 4"; return false; }
    if ((g.pitch_j * es) % 16 || (g.pitch_k * es) % 16) { *why = "pitches are not multiples of 16 bytes"; return false; }
    const long long r = g.origin - (long long)(g.halo - 1) * g.pitch_j;
    if (r < 0 || r >= g.pitch_j) { *why = "origin is not within the first padded row"; return false; }
    if ((r + 1) % padx) { *why = "interior rows do not start on a 16-byte boundary"; return false; }
    if (r + g.nx + g.halo + 1 > g.pitch_j) { *why = "row does not fit its pitch"; return false; }
    if (g.nz + 2 > (1 << 30) || g.ny + 2 * g.halo > (1 << 30)) { *why = "grid too large for a tensor map"; return false; }
    *ox_out = (int)r;
    return true;
}

bool pw::aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Device (or managed) memory of `device`?  A host address handed to a kernel
// would fault the GPU, so every field pointer is checked on the host first.
bool pw::is_device_ptr(const void* p, int device) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();   // clear the sticky-free error of the query
        return false;
    }
    if (a.type == cudaMemoryTypeManaged) return true;
    return a.type == cudaMemoryTypeDevice && a.device == device;
}

// The entry of a handle's cache of recently encoded maps for these cells of a
// field and this box, its map encoded by `encode` (a status) if it is not there.
template <class Encode>
static pw_status_t cached_map(pw_handle_t h, const void* ptr, int kind, int box_w, int box_h, CUtensorMap* out,
                              const Encode& encode) {
    for (auto& c : h->maps)
        if (c.ptr == ptr && c.kind == kind && c.box_w == box_w && c.box_h == box_h) {
            *out = c.map;
            return PW_OK;
        }
    const pw_status_t st = encode();
    if (st != PW_OK) return st;
    MapCacheEntry& e = h->maps[h->map_next];
    h->map_next = (h->map_next + 1) % (int)(sizeof(h->maps) / sizeof(h->maps[0]));
    e.ptr = ptr;
    e.kind = kind;
    e.box_w = box_w;
    e.box_h = box_h;
    e.map = *out;
    return PW_OK;
}

static pw_status_t encode_map_box(pw_handle_t h, const void* ptr, int box_w, int box_h, CUtensorMap* out) {
    return cached_map(h, ptr, MAP_FIELD, box_w, box_h, out,
                      [&] { return encode_tensor_map_box(h->grid, ptr, box_w, box_h, out); });
}

// Tensor map for a launch shape of the single-grid k-march.
static pw_status_t encode_map(pw_handle_t h, const void* ptr, const TmaConfig& c, CUtensorMap* out) {
    if (c.rag == 2) {
        const PackedRows p = packed_rows(h->grid.nx, (int)dtype_size(h->grid.dtype));
        return encode_map_box(h, ptr, p.box_w, p.rows + 2, out);
    }
    return encode_map_box(h, ptr, tma_box_width(h->grid.dtype, c.lx, c.nc), c.ty + 2, out);
}

pw_status_t pw::encode_tensor_map(const pw_grid_t& g, const void* ptr, int lx, int ty, CUtensorMap* out, int nc,
                                  int l2_promotion) {
    return encode_tensor_map_box(g, ptr, tma_box_width(g.dtype, lx, nc), ty + 2, out, l2_promotion);
}

// 3D map of one field: x = the padded row from its first element (element
// i = 0 at x = ox), y = rows from j = 1-halo, z = levels 0..nz+1.  Boxes of
// box_w x box_h x 1; out-of-range elements read as zero.
pw_status_t pw::encode_tensor_map_box(const pw_grid_t& g, const void* ptr, int box_w, int box_h, CUtensorMap* out,
                                      int l2_promotion) {
    int ox = 0;
    const char* why = "";
    // (the callers decide about widths: a box may run past the row's end)
    if (!tma_layout_ok(g, &ox, &why, true)) return fail(PW_ERR_UNSUPPORTED, "layout not TMA-eligible: %s", why);
    return encode_tensor_map_dims(g, ptr, {ox + g.nx + g.halo + 1, g.ny + 2 * g.halo, g.nz + 2}, box_w, box_h, out,
                                  l2_promotion);
}

pw_status_t pw::encode_tensor_map_dims(const pw_grid_t& g, const void* base, const long long (&n)[3], int box_w,
                                       int box_h, CUtensorMap* out, int l2_promotion) {
    auto fn = encode_fn();
    if (!fn) return fail(PW_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    if (inject_failure(INJECT_TENSOR_MAP)) return fail(PW_ERR_CUDA, "cuTensorMapEncodeTiled failed (injected)");
    const size_t es = dtype_size(g.dtype);
    CUtensorMapDataType dt = g.dtype == PW_F32    ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                             : g.dtype == PW_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                  : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    cuuint64_t dims[3] = {(cuuint64_t)n[0], (cuuint64_t)n[1], (cuuint64_t)n[2]};
    cuuint64_t strides[2] = {(cuuint64_t)(g.pitch_j * es), (cuuint64_t)(g.pitch_k * es)};
    cuuint32_t box[3] = {(cuuint32_t)box_w, (cuuint32_t)box_h, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(out, dt, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_NONE, (CUtensorMapL2promotion)l2_promotion,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(PW_ERR_CUDA, "cuTensorMapEncodeTiled failed (CUresult %d)", (int)r);
    return PW_OK;
}

// A tensor map of the TMA adjoint for field f of (u, v, w, lsu, lsv, lsw), and
// where levels, rows and columns lie in such maps (AdjGeom).  u, v, w: levels
// 1..nz of whole rows with their halos, or (open mode) of columns -3..nx+1 (-3 is
// the first 16-byte boundary at or before column 0; interior rows start on one)
// and rows 0..ny+1.  Sensitivities: levels 2..nz (lsw 2..nz-1) of whole rows with
// their halos, or (the modes that do not read these) of the interior.
static AdjGeom adj_geom(const pw_grid_t& g, int ox, AdjMode mode) {
    if (mode == ADJ_OPEN) return AdjGeom{3, 0, -1, -1, -1, -2, -3, 0, 0, g.nx + 1, 0, g.ny + 1};
    if (mode == ADJ_PERIODIC_ANY)
        return AdjGeom{ox, g.halo - 1, -1, -1, -1, -2, 1, 1, 2, g.nx - 1, 2, g.ny - 1};
    return AdjGeom{ox, g.halo - 1, -1, ox, g.halo - 1, -2, 1, 1, 1, g.nx, 1, g.ny};
}
static pw_status_t adj_map(pw_handle_t h, int f, const void* ptr, AdjMode mode, int ox, int box_w, int box_h,
                           CUtensorMap* out) {
    const int kind = MAP_ADJ + 3 * (f < 3 ? 0 : (f < 5 ? 1 : 2)) + (int)mode;
    const pw_grid_t& g = h->grid;
    const AdjGeom ge = adj_geom(g, ox, mode);
    // the map's first element: level, row and column with coordinate 0
    const long long k = f < 3 ? -ge.fz : -ge.lz, j = f < 3 ? -ge.fy : -ge.ly, i = f < 3 ? -ge.fx : -ge.lx;
    const float* base = static_cast<const float*>(ptr) + g.origin + k * g.pitch_k + j * g.pitch_j + i;
    const long long levels = f < 3 ? g.nz : (f < 5 ? g.nz - 1 : g.nz - 2);
    const bool whole = mode == ADJ_PERIODIC || (mode == ADJ_PERIODIC_ANY && f < 3);
    const long long rows = whole ? g.ny + 2LL * g.halo : (f < 3 ? g.ny + 2 : g.ny);
    const long long cols = whole ? ox + g.nx + g.halo + 1LL : (f < 3 ? g.nx + 5 : g.nx);
    return cached_map(h, ptr, kind, box_w, box_h, out,
                      [&] { return encode_tensor_map_dims(g, base, {cols, rows, levels}, box_w, box_h, out); });
}

// Every pointer in ps[0..n) is device memory of the handle's GPU (checked
// once per pointer, then remembered).
static pw_status_t check_device_ptrs(pw_handle_t h, const void* const* ps, int n) {
    for (int a = 0; a < n; ++a) {
        const void* p = ps[a];
        bool known = false;
        for (auto q : h->dev_ok) known = known || (q == p);
        if (known) continue;
        if (!is_device_ptr(p, h->device))
            return fail(PW_ERR_ARG, "field pointer %p is not device memory of GPU %d", p, h->device);
        h->dev_ok[h->dev_next] = p;
        h->dev_next = (h->dev_next + 1) % pw_handle_s::kDevCache;
    }
    return PW_OK;
}

// Launch shape of the TMA kernel for the source terms (step = false) or the
// fused step (step = true).  A shape the user fixed (pw_set_tma_config) is used
// as given, unset fields at the scalar defaults (32 lanes x 4 cells x 4 rows, 4
// stages, one row per thread).  Otherwise 4 stages and one of these (lanes x
// cells x rows), with the k segments, whichever march_cost puts lowest:
//   narrow, no multiple of 4:   packed rows alone (kPackedNx);
//   nx <= 64:                   16 x 4 x 4 alone;
//   FP32:                       32 x 4 x 4, 16 x 4 x 8, 8 x 4 x 16;
//   16-bit (source terms; steps when nx % 8 = 0):
//                               16 x 8 x 8, 8 x 8 x 16, a thread's cells
//                               packed as FP32x2 pairs along x;
//   16-bit steps otherwise:     32 x 4 x 4, 16 x 4 x 8 in x pairs (the 8-cell
//                               form spills with ragged rows: 335 us a step
//                               against 218 at 1021 x 1023 x 61).
// The first of each line is the fastest on whole tiles; the narrower ones cover
// fewer cells beyond nx.  FP32 source terms, first shape alone against the
// choice: 160x824x41 39.2 -> 29.1 us, 184x1280x21 33.6 -> 27.6, 776x184x29 25.4
// -> 21.3, 320x1120x26 48.0 -> 45.5; BF16 320x1216x69 94.9 -> 82.8, 1056x1552x24
// 122 -> 115, 512x512x64 (segments alone) 61 -> 55.  Grids below kShapeMinCells
// keep the first shape: a call of that size is launch and latency.
constexpr long long kShapeMinCells = 1 << 18;
constexpr int kMaxGridY = 65535;   // CTAs of a launch along y (and z)

// Widths that are no multiple of 4 run in packed rows (PackedRows) up to these
// columns.  Beyond, a row leaves threads idle (21 vectors: 126 of 128, 22: 110)
// and the tiles fit better: FP32 source terms, packed / tiles, 69 x 787 x 89 32.3 /
// 34.0 us, 79 x 203 x 69 9.9 / 9.9, 83 x 223 x 51 8.9 / 8.5; 16-bit ones and steps,
// whose tiles are 64 columns wide, 83 x 223 x 51 8.8 / 9.5 and 11.7 / 14.5, 114 x 453
// x 82 26.9 / 21.1 and 42.0 / 35.7.
constexpr int kPackedNx = 80, kPackedNx16 = 96;

// Estimated time of a march in units of one level of a full SM: `slots` CTAs
// fit the GPU, each marches its levels after a start that costs as much as 1.6
// of them (x pairs, whose levels take longer: 0.8); a last wave that leaves SMs
// with r of their R slots takes 0.7 + 0.3 r / R of a full one (x pairs: 0.45 +
// 0.55 r / R), as fewer CTAs on an SM each run faster.  Fitted to a sweep of
// shapes and segments over 31 grids (64^3 to 1056 x 1552 x 24): in the mean the
// choice is within 1 % (FP32 source terms), 2 % (16-bit), 3 to 4 % (steps) of
// the sweep's best, where counting whole waves of (levels + 2) was 8 % off.
// FP32 steps, after a sweep over 135 grids from 2e4 to 4e7 cells: 0.3 of a wave
// more where the fields exceed L2 (kL2Cells), 0.4 for grids at most 64 columns wide:
// the time in which the first and last CTAs leave the memory idle.  Without it one
// wave of whole columns looks too cheap there (652 x 449 x 55: one segment 101 us, four
// 86, 8-lane tiles in seven 80; 56 x 1088 x 84: five 48, eight 42).  The choice is then
// within 1.2 % of the sweep's best in the mean.
constexpr long long kL2Cells = 6000000;   // 24 bytes each: a little more than L2
static long long march_tiles(const pw_grid_t& gr, const TmaConfig& c) {
    const int rows = c.rag == 2 ? packed_rows(gr.nx, (int)dtype_size(gr.dtype)).rows : c.ty;
    return (c.rag == 2 ? 1LL : (gr.nx + c.nc * c.lx - 1) / (c.nc * c.lx)) * ((gr.ny + rows - 1) / rows);
}
static double march_cost(const pw_grid_t& gr, const TmaConfig& c, bool step, int n, int sms, int bps) {
    const long long ctas = march_tiles(gr, c) * n, slots = (long long)sms * bps;
    const long long full = ctas / slots, rem = ctas - full * slots;
    const double w = c.xp ? 0.45 : 0.7;
    double out = 0.0;
    if (step && gr.dtype == PW_F32 && !c.rag)
        out = gr.nx <= 64 ? 0.4 : ((long long)gr.nx * gr.ny * gr.nz > kL2Cells ? 0.3 : 0.0);
    const double last = rem ? w + (1.0 - w) * (double)((rem + sms - 1) / sms) / bps : 0.0;
    return ((gr.nz + n - 1) / n + (c.xp ? 0.8 : 1.6)) * ((double)full + last + out) * bps * (c.nc * c.lx) * c.ty;
}

static TmaConfig choose_tma(pw_handle_t h, bool step) {
    TmaConfig& cache = h->tma_auto[step ? 1 : 0];
    if (cache.ty) return cache;
    const TmaConfig& u = h->tma_user;
    const pw_grid_t& gr = h->grid;
    TmaConfig cand[4];
    int nc = 0;
    auto add = [&](int lx, int cells, int ty, int xp, int rp) {
        TmaConfig c{lx, ty, 4, 1, cells};
        c.rp = rp;
        c.xp = xp;
        cand[nc++] = c;
    };
    if (u.lx || u.nc || u.ty || u.stages || u.rp) {   // rows_per_thread 3: one row, cells paired along x
        add(u.lx ? u.lx : 32, u.nc ? u.nc : 4, u.ty ? u.ty : 4, u.rp == 3, (u.rp && u.rp != 3) ? u.rp : 1);
        if (u.stages) cand[0].stages = u.stages;
    } else {
        const bool half = dtype_size(gr.dtype) == 2, more = (long long)gr.nx * gr.ny * gr.nz >= kShapeMinCells;
        const bool packed = gr.nx % 4 && gr.nx <= (half ? kPackedNx16 : kPackedNx);
        if (packed) {
            add(32, 4, 4, 0, 1);
        } else if (gr.nx <= 64) {
            add(16, 4, 4, 0, 1);
        } else if (!half) {
            add(32, 4, 4, 0, 1);
            if (step && gr.nx % 4 == 0) cand[0].few = 1;
            if (cand[0].few && more) add(32, 4, 4, 0, 1);
            if (more) add(16, 4, 8, 0, 1);
            if (more) add(8, 4, 16, 0, 1);
        } else if (!step || gr.nx % 8 == 0) {
            add(16, 8, 8, 1, 1);
            if (more) add(8, 8, 16, 1, 1);
        } else {
            add(32, 4, 4, 1, 1);
            if (more) add(16, 4, 8, 1, 1);
        }
        for (int q = 0; q < nc; ++q) cand[q].rag = gr.nx % 4 ? (packed ? 2 : 1) : 0;
        if (step && gr.nx % 4 == 0 && gr.nx < 64)   // (see tma_min_blocks)
            cand[0].few = (long long)gr.nx * gr.ny * gr.nz < (1 << 17);
    }
    TmaConfig best = cand[0];
    double lowest = 0.0;
    for (int q = 0; q < nc; ++q) {
        TmaConfig c = cand[q];
        int bps = step ? step_blocks_per_sm(gr.dtype, c) : tma_blocks_per_sm(gr.dtype, c);
        if (bps < 1) bps = 1;
        const int lo = u.nseg ? u.nseg : 1, hi = u.nseg ? u.nseg : std::max(1, gr.nz / 2);
        for (c.nseg = lo; c.nseg <= hi; ++c.nseg) {
            if (c.few && nc > 1 && march_tiles(gr, c) * c.nseg > (long long)h->num_sms * bps) break;
            const double cost = march_cost(gr, c, step, c.nseg, h->num_sms, bps);
            if (lowest > 0.0 && !(cost < 0.985 * lowest)) continue;   // narrower or more segments only for a gain
            lowest = cost;
            best = c;
        }
    }
    if (best.nseg > gr.nz / 2) best.nseg = std::max(1, gr.nz / 2);
    cache = best;
    return best;
}

// TMA k-march or generic kernel for the source terms and the steps: what
// pw_set_kernel asked for, else TMA when the layout and every pointer qualify.
// A width that is no multiple of 4 takes the k-march too (its RAG kernels) when
// the shape is automatic and the grid has at least kRagMinCells cells; FP32
// steps on tiles that cover more than 1.1 x the width (packed rows aside) from
// kRagMinStepCells cells.  Measured on GB300, generic against k-march, us:
//   source terms  FP32 41x168x69 (475 k cells) 6.6 / 7.0, 33x1000x16 6.8 / 6.6, 131x66x61 7.0 / 6.5, 229x57x47
//                 7.8 / 7.2, 39x785x49 16.9 / 12.7, 511x256x64 111 / 44.5, 1021x1023x61 943 / 259; BF16 33x1000x16
//                 7.0 / 6.8, 131x66x61 7.4 / 7.7, 511x64x17 7.2 / 6.8, 69x787x89 60.9 / 28.8;
//   a step        FP32 33x129x125 (532 k) 8.2 / 9.2, 34x250x62 8.1 / 8.2, 65x129x64 8.0 / 7.9, 386x35x49 (662 k) 9.1 /
//                 8.2, 39x785x49 20.7 / 17.0, 511x256x64 119 / 62; on tiles that fit badly 97x129x64 10.4 / 11.3,
//                 102x489x17 10.5 / 13.2, 137x389x25 15.4 / 17.0, 135x129x128 (2.2 M) 25.7 / 24.4; BF16 33x1000x16
//                 8.4 / 9.5, 97x129x64 11.3 / 11.1, 66x129x125 14.6 / 12.2, 39x785x49 19.3 / 16.8.
// Below kRagMinNx columns the generic kernel stays: 9x2048x77 38.3 / 38.9, 17x2048x17 7.6 / 9.3, 13x1265x84 26.6 /
// 21.3.  pw_set_kernel(2) refuses such a width as it always has.
constexpr int kRagMinNx = 32;
constexpr long long kRagMinCells = 1 << 19, kRagMinStepCells = 1 << 21;
static bool ragged_on_march(pw_handle_t h, bool step) {
    const TmaConfig& u = h->tma_user;
    const pw_grid_t& gr = h->grid;
    const long long cells = (long long)gr.nx * gr.ny * gr.nz;
    if (h->kernel_kind != 0 || gr.nx < kRagMinNx || cells < kRagMinCells || u.lx || u.nc || u.ty || u.stages || u.rp)
        return false;
    const bool packed = gr.nx <= (gr.dtype == PW_F32 ? kPackedNx : kPackedNx16);
    if (!packed && step && gr.dtype == PW_F32 && cells < kRagMinStepCells &&
        10LL * ((gr.nx + 31) / 32 * 32) > 11LL * gr.nx)
        return false;
    const int rows = packed ? packed_rows(gr.nx, (int)dtype_size(gr.dtype)).rows : 4;   // the lowest tile's
    return gr.ny <= (long long)kMaxGridY * rows;
}
static pw_status_t march_kernel_choice(pw_handle_t h, bool step, const void* const* bufs, int n, bool* use_tma,
                                       int* ox) {
    const char* why = "";
    const bool any_nx = h->grid.nx % 4 && ragged_on_march(h, step);
    const bool layout_ok = tma_layout_ok(h->grid, ox, &why, any_nx);
    bool ptrs_ok = true;
    for (int a = 0; a < n; ++a) ptrs_ok = ptrs_ok && aligned16(bufs[a]);
    if (h->kernel_kind == 2) {
        if (!layout_ok) return fail(PW_ERR_UNSUPPORTED, "TMA kernel requested but %s", why);
        if (!ptrs_ok) return fail(PW_ERR_ALIGN, "TMA kernel requested but a field pointer is not 16-byte aligned");
    }
    *use_tma = (h->kernel_kind == 2) || (h->kernel_kind == 0 && layout_ok && ptrs_ok);
    return PW_OK;
}

static void make_scales(const float* scale, Scales* sc, bool* scaled) {
    *scaled = false;
    for (int q = 0; q < 3; ++q) {
        sc->in[q] = scale ? scale[q] : 1.f;
        sc->out[q] = scale ? scale[3 + q] : 1.f;
        if (sc->in[q] != 1.f || sc->out[q] != 1.f) *scaled = true;
    }
}

namespace pw {

pw_status_t internal_fail(pw_status_t s, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return s;
}

pw_status_t internal_cuda_fail(cudaError_t e, const char* what) { return cuda_fail(e, what); }

static std::atomic<int> g_inject[INJECT_KINDS];

bool inject_failure(int kind) {
    int n = g_inject[kind].load(std::memory_order_relaxed);
    while (n > 0)
        if (g_inject[kind].compare_exchange_weak(n, n - 1, std::memory_order_relaxed)) return true;
    return false;
}

cudaError_t set_smem_attr_once_impl(const void* kern, int bytes) {
    static std::mutex mu;
    static std::vector<std::pair<const void*, int>> done;   // (kernel, device)
    static thread_local std::pair<const void*, int> last{nullptr, -1};   // this thread's last one found done
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (last.first == kern && last.second == dev) return cudaSuccess;
    std::lock_guard<std::mutex> lock(mu);
    for (auto& d : done)
        if (d.first == kern && d.second == dev) {
            last = d;
            return cudaSuccess;
        }
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    // all the shared memory an SM has, so that shared memory does not hold the
    // resident CTAs below what the registers allow (the kernels stage their
    // data in shared memory and barely use the L1 cache)
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) done.emplace_back(kern, dev);
    return e;
}

bool internal_handle_grid(pw_handle_t h, pw_grid_t* g, int* num_sms) {
    if (!h) return false;
    *g = h->grid;
    *num_sms = h->num_sms;
    return true;
}

int internal_handle_device(pw_handle_t h) { return h ? h->device : -1; }

pw_status_t internal_check_device_ptrs(pw_handle_t h, const void* const* ps, int n) {
    return check_device_ptrs(h, ps, n);
}

}  // namespace pw

extern "C" {

pw_status_t pw_grid_default(int32_t nx, int32_t ny, int32_t nz, int32_t halo, pw_dtype_t dtype, pw_grid_t* out,
                            int64_t* alloc_elems) {
    if (!out) return fail(PW_ERR_ARG, "out is NULL");
    if (dtype != PW_F32 && dtype != PW_BF16 && dtype != PW_F16) return fail(PW_ERR_ARG, "unknown dtype");
    if (nx < 1 || ny < 1 || nz < 3 || halo < 1) return fail(PW_ERR_ARG, "need nx, ny >= 1, nz >= 3, halo >= 1");
    const long long line = 128 / (long long)dtype_size(dtype);   // elements per 128 bytes
    // interior i = 1 at x = ox + 1, a multiple of `line`, with room for the halo
    const long long ox = ((halo + line - 1) / line) * line - 1;
    const long long pj = ((ox + 1 + nx + halo + line - 1) / line) * line;
    const long long pk = pj * (ny + 2LL * halo);
    pw_grid_t g;
    g.nx = nx;
    g.ny = ny;
    g.nz = nz;
    g.halo = halo;
    g.pitch_j = pj;
    g.pitch_k = pk;
    g.origin = ox + (long long)(halo - 1) * pj;
    g.dtype = dtype;
    *out = g;
    if (alloc_elems) *alloc_elems = pk * (nz + 2LL);
    return PW_OK;
}

pw_status_t pw_create(const pw_grid_t* grid, const pw_coeffs_t* coeffs, pw_handle_t* out) {
    if (!out) return fail(PW_ERR_ARG, "out is NULL");
    *out = nullptr;
    pw_status_t s = validate_grid(grid);
    if (s != PW_OK) return s;
    if (!coeffs || !coeffs->tzc1 || !coeffs->tzc2 || !coeffs->tzd1 || !coeffs->tzd2)
        return fail(PW_ERR_ARG, "coefficients or one of the vertical coefficient arrays is NULL");
    pw_handle_s* h = new (std::nothrow) pw_handle_s();
    if (!h) return fail(PW_ERR_OOM, "host allocation of the handle failed");
    h->grid = *grid;
    h->tcx = (float)coeffs->tcx;
    h->tcy = (float)coeffs->tcy;
    cudaError_t e = cudaGetDevice(&h->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
    const int n = grid->nz + 2;
    std::vector<float> tz(4 * (size_t)n);
    for (int k = 0; k < n; ++k) {
        tz[k] = (float)coeffs->tzc1[k];
        tz[n + k] = (float)coeffs->tzc2[k];
        tz[2 * n + k] = (float)coeffs->tzd1[k];
        tz[3 * n + k] = (float)coeffs->tzd2[k];
    }
    if (e == cudaSuccess) e = dev_malloc(&h->d_tz, tz.size() * sizeof(float));
    if (e == cudaSuccess) e = cudaMemcpy(h->d_tz, tz.data(), tz.size() * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = dev_malloc(&h->d_err, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(h->d_err, 0, sizeof(int));
    // the upload and the clear run on the legacy default stream, which the
    // caller's non-blocking streams do not wait for: finish them here
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    if (e != cudaSuccess) {
        pw_destroy(h);
        return cuda_fail(e, "pw_create");
    }
    *out = h;
    return PW_OK;
}

pw_status_t pw_destroy(pw_handle_t h) {
    if (!h) return PW_OK;
    for (auto& st : h->hs)   // an asynchronous host call may still be running
        if (st) cudaStreamSynchronize(st);
    for (auto& st : h->hs)
        if (st) cudaStreamDestroy(st);
    for (int c = 0; c < pw_handle_s::kMaxChunks; ++c) {
        if (h->ev_in[c]) cudaEventDestroy(h->ev_in[c]);
        if (h->ev_comp[c]) cudaEventDestroy(h->ev_comp[c]);
        if (h->ev_out[c]) cudaEventDestroy(h->ev_out[c]);
    }
    if (h->ev_start) cudaEventDestroy(h->ev_start);
    if (h->ev_end) cudaEventDestroy(h->ev_end);
    cudaFree(h->d_tz);
    cudaFree(h->d_err);
    for (auto& p : h->d_stage) cudaFree(p);
    cudaFree(h->d_scratch);
    delete h;
    return PW_OK;
}

pw_status_t pw_set_kernel(pw_handle_t h, int32_t kind) {
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (kind < 0 || kind > 2) return fail(PW_ERR_ARG, "kernel kind must be 0, 1 or 2");
    h->kernel_kind = kind;
    return PW_OK;
}

pw_status_t pw_set_tma_config(pw_handle_t h, int32_t lanes_x, int32_t cells, int32_t ty, int32_t stages,
                              int32_t nseg, int32_t rows_per_thread) {
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (nseg < 0 || nseg > h->grid.nz / 2) return fail(PW_ERR_ARG, "nseg must be in 0..nz/2");
    if (rows_per_thread < 0 || rows_per_thread > 3)
        return fail(PW_ERR_ARG, "rows_per_thread must be 0, 1, 2 or 3");
    TmaConfig c{lanes_x ? lanes_x : 32, ty ? ty : 4, stages ? stages : 4, 1};
    c.nc = cells ? cells : 4;
    c.rp = rows_per_thread ? rows_per_thread : 1;
    if (c.rp == 3) {
        c.rp = 1;
        c.xp = 1;
    }
    if (!tma_config_supported(h->grid.dtype, c))
        return fail(PW_ERR_UNSUPPORTED,
                    "no TMA kernel instance for lanes_x=%d cells=%d ty=%d stages=%d rows_per_thread=%d (dtype %d)",
                    c.lx, c.nc, c.ty, c.stages, rows_per_thread ? rows_per_thread : 1, (int)h->grid.dtype);
    h->tma_user = TmaConfig{lanes_x, ty, stages, nseg};
    h->tma_user.nc = cells;
    h->tma_user.rp = rows_per_thread;
    h->tma_auto[0] = h->tma_auto[1] = TmaConfig{0, 0, 0, 0};
    for (auto& m : h->maps) m.ptr = nullptr;
    return PW_OK;
}

pw_status_t pw_set_step_blocking(pw_handle_t h, int32_t steps_per_pass, int32_t ty, int32_t stages,
                                 int32_t ctas_per_sm, int32_t nseg) {
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (steps_per_pass < 0 || steps_per_pass > 2) return fail(PW_ERR_ARG, "steps_per_pass must be 0, 1 or 2");
    if (nseg < 0 || nseg > h->grid.nz / 2) return fail(PW_ERR_ARG, "nseg must be in 0..nz/2");
    Step2Config c{ty ? ty : 16, stages ? stages : 3, 1, ctas_per_sm ? ctas_per_sm : 1};
    if (!step2_config_supported(c))
        return fail(PW_ERR_UNSUPPORTED, "no two-step kernel instance for ty=%d stages=%d ctas_per_sm=%d", c.ty,
                    c.stages, c.minb);
    h->steps_per_pass = steps_per_pass;
    h->step2_user = Step2Config{ty, stages, nseg, ctas_per_sm};
    h->step2_auto = Step2Config{0, 0, 0, 0};
    return PW_OK;
}

// Launch shape of the two-step kernel: user overrides, else 16 rows, 3 stages,
// one CTA of 16 warps per SM (the fastest measured on GB300, 2048^2 x 64:
// FP32 208, BF16 201 Gcell-steps/s, against 156 and 152 with 8 rows), and k
// segments doubled until about two waves of CTAs cover the SMs (each segment
// keeps >= 8 levels).
static Step2Config choose_step2(pw_handle_t h) {
    if (h->step2_auto.ty) return h->step2_auto;
    const Step2Config& u = h->step2_user;
    Step2Config c{u.ty ? u.ty : 16, u.stages ? u.stages : 3, 1, u.minb ? u.minb : 1};
    if (u.nseg) {
        c.nseg = u.nseg;
    } else {
        const long long tiles = (long long)((h->grid.nx + step2_tile_cols() - 1) / step2_tile_cols()) *
                                ((h->grid.ny + c.ty - 3) / (c.ty - 2));
        int bps = step2_blocks_per_sm(h->grid.dtype, c);
        if (bps < 1) bps = 1;
        const long long slots = (long long)h->num_sms * bps;
        int nseg = 1;
        while (tiles * nseg < 2 * slots && h->grid.nz / (nseg * 2) >= 8) nseg *= 2;
        c.nseg = nseg;
    }
    if (c.nseg > h->grid.nz / 2) c.nseg = std::max(1, h->grid.nz / 2);
    h->step2_auto = c;
    return c;
}

// The caller fixed a shape that only the periodic mode of widths that are a
// multiple of 4 is instantiated for.
static bool adj_fixed(pw_handle_t h) {
    const AdjConfig& u = h->adj_user;
    return (u.na || u.ty || u.stages) && adjoint_shape(u).lx != 16;
}

// Launch shape of the TMA adjoint (periodic or open mode): each field the user
// fixed, else 32 lanes x 4 cells x 6 rows with 4 slots for periodic grids below
// kShapeMinCells, and 16 lanes x 4 cells x 8 rows with 3 slots otherwise; k
// segments (automatic) of >= 4 levels, the count with the lowest estimated
// time as for the k-march, a segment's start costing 2.5 levels (two planes
// more than its levels, the priming level).  Periodic small grids, (4, 6, 4) / (4,
// 8, 3) in us: 64x8x4 8.2 / 8.9, 32x32x32 8.9 / 8.6, 64x64x32 8.9 / 8.7, 128x64x30
// 10.1 / 9.6, 64x64x64 10.3 / 9.4.  The full array has (4, 8, 3) alone, against the
// gather kernel 8x8x8 7.2 / 20.5, 32x32x16 7.9 / 18.8, 64x64x64 9.8 / 44.6; odd periodic
// widths 127x64x40 26.8 / 30.6, 33x250x60 35.8 / 48.6.
static AdjConfig choose_adjoint(pw_handle_t h, AdjMode mode) {
    AdjConfig& cache = h->adj_auto[mode];
    if (cache.na) return cache;
    const AdjConfig& u = h->adj_user;
    const pw_grid_t& gr = h->grid;
    AdjConfig c = adjoint_shape(u);
    if (mode != ADJ_PERIODIC || (!u.na && !u.ty && !u.stages && (long long)gr.nx * gr.ny * gr.nz >= kShapeMinCells))
        c = AdjConfig{4, 8, 3, u.nseg, 16};
    if (!c.nseg) {
        const AdjGeom ge = adj_geom(gr, 0, mode);
        const int wx = std::max(1, ge.ihi - ge.i0 + 1), wy = std::max(1, ge.jhi - ge.j0 + 1), tx = c.lx * c.na;
        const long long tiles = (long long)((wx + tx - 1) / tx) * ((wy + c.ty - 1) / c.ty);
        const int bps = std::max(1, adjoint_blocks_per_sm(c, mode != ADJ_PERIODIC));
        const long long slots = (long long)h->num_sms * bps;
        double lowest = 0.0;
        for (int n = 1; n == 1 || gr.nz / n >= 4; ++n) {
            const long long full = tiles * n / slots, rem = tiles * n - full * slots;
            const double last = rem ? 0.6 + 0.4 * (double)((rem + h->num_sms - 1) / h->num_sms) / bps : 0.0;
            const double cost = ((gr.nz + n - 1) / n + 2.5) * ((double)full + last);
            if (lowest > 0.0 && !(cost < 0.985 * lowest)) continue;
            lowest = cost;
            c.nseg = n;
        }
    }
    const int most = mode == ADJ_PERIODIC ? kAdjMaxSeg : kAdjMaxSegChecked;
    c.nseg = std::min(std::max(c.nseg, (gr.nz + most - 1) / most), (int)gr.nz);
    cache = c;
    return c;
}

pw_status_t pw_set_adjoint_config(pw_handle_t h, int32_t cells, int32_t ty, int32_t stages, int32_t nseg) {
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (cells < 0 || ty < 0 || stages < 0) return fail(PW_ERR_ARG, "cells, ty and stages must be >= 0");
    if (nseg < 0 || nseg > h->grid.nz) return fail(PW_ERR_ARG, "nseg must be in 0..nz");
    const AdjConfig c = adjoint_shape(AdjConfig{cells, ty, stages, nseg});
    if (!adjoint_config_supported(c))
        return fail(PW_ERR_UNSUPPORTED, "no TMA adjoint instance for cells=%d ty=%d stages=%d", c.na, c.ty,
                    c.stages);
    h->adj_user = AdjConfig{cells, ty, stages, nseg};
    for (auto& a : h->adj_auto) a = AdjConfig{};
    return PW_OK;
}

pw_status_t pw_get_adjoint_config(pw_handle_t h, int32_t out[4]) {
    if (!h || !out) return fail(PW_ERR_ARG, "handle or out is NULL");
    const AdjConfig c = choose_adjoint(h, h->grid.nx % 4 && !adj_fixed(h) ? ADJ_PERIODIC_ANY : ADJ_PERIODIC);
    out[0] = c.na;
    out[1] = c.ty;
    out[2] = c.stages;
    out[3] = c.nseg;
    return PW_OK;
}

pw_status_t pw_get_tma_config(pw_handle_t h, int32_t step, int32_t out[6]) {
    if (!h || !out) return fail(PW_ERR_ARG, "handle or out is NULL");
    const TmaConfig c = choose_tma(h, step != 0);
    const PackedRows p = packed_rows(h->grid.nx, (int)dtype_size(h->grid.dtype));
    out[0] = c.rag == 2 ? p.vec : c.lx;
    out[1] = c.nc;
    out[2] = c.rag == 2 ? p.rows : c.ty;
    out[3] = c.stages;
    out[4] = c.nseg;
    out[5] = c.xp ? 3 : c.rp;
    return PW_OK;
}

int32_t pw_last_kernel(pw_handle_t h) { return h ? h->last_kernel : 0; }

pw_status_t pw_tendencies(pw_handle_t h, const void* u, const void* v, const void* w, void* su, void* sv,
                          void* sw, const float* scale, pw_stream_t stream) {
    PW_RANGE("pw_tendencies");
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (!u || !v || !w || !su || !sv || !sw) return fail(PW_ERR_ARG, "a field pointer is NULL");
    const void* ins[3] = {u, v, w};
    const void* outs[3] = {su, sv, sw};
    for (auto o : outs)
        for (auto i : ins)
            if (o == i) return fail(PW_ERR_ARG, "an output aliases an input");
    if (su == sv || su == sw || sv == sw) return fail(PW_ERR_ARG, "outputs alias each other");
    {
        const void* ptrs[6] = {u, v, w, su, sv, sw};
        pw_status_t dst = check_device_ptrs(h, ptrs, 6);
        if (dst != PW_OK) return dst;
    }
    if (scale)
        for (int q = 0; q < 6; ++q)
            if (!(scale[q] > 0.f) || !(scale[q] < 3.0e38f)) return fail(PW_ERR_ARG, "scales must be finite and > 0");
    Scales sc;
    bool scaled;
    make_scales(scale, &sc, &scaled);
    const GridDev g = to_dev(h->grid);
    CoefDev cf{h->tcx, h->tcy, h->d_tz};
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);

    int ox = 0;
    const void* all[6] = {u, v, w, su, sv, sw};
    bool use_tma = false;
    pw_status_t kst = march_kernel_choice(h, false, all, 6, &use_tma, &ox);
    if (kst != PW_OK) return kst;
    if (use_tma) {
        TmaConfig c = choose_tma(h, false);
        CUtensorMap maps[3];
        for (int q = 0; q < 3; ++q) {
            pw_status_t st = encode_map(h, ins[q], c, &maps[q]);
            if (st != PW_OK) return st;
        }
        cudaError_t e = launch_tend_tma(h->grid.dtype, g, ox, maps, su, sv, sw, sc, cf, h->d_err, c, s);
        if (e != cudaSuccess) return cuda_fail(e, "TMA tendency kernel launch");
        h->last_kernel = 2;
    } else {
        cudaError_t e = launch_tend_generic(h->grid.dtype, g, u, v, w, su, sv, sw, sc, scaled, cf, h->num_sms, s);
        if (e != cudaSuccess) return cuda_fail(e, "generic tendency kernel launch");
        h->last_kernel = 1;
    }
    return PW_OK;
}

// Levels per chunk of the host path's copy / compute pipeline (build knob).
// The first chunk's copy in and the last chunk's copy out run alone, so
// smaller chunks overlap more; measured on GB300 (2048^2 x 64 FP32, pitched
// box copies): 16 levels 11.8, 8: 12.5-12.7, 4: 13.0-13.1, 2: 13.1 Gcell/s.
#ifndef PW_HOST_CHUNK_LEVELS
#define PW_HOST_CHUNK_LEVELS 4
#endif

// Copy the box i0..i0+ni-1, j0..j0+nj-1, levels k0..k1 of a field between
// host and device buffers of the same layout: one 3D copy when a level is a
// whole number of rows, else one 2D copy per level.  Only the box travels
// (no row padding, no rows or columns outside it).
static cudaError_t copy_box(const pw_grid_t& g, void* dst, const void* src, int i0, int ni, int j0, int nj, int k0,
                            int k1, cudaMemcpyKind kind, cudaStream_t s) {
    const size_t es = dtype_size(g.dtype);
    const size_t pitch = (size_t)g.pitch_j * es;
    auto at = [&](const void* base, int k) {
        return (char*)base + (size_t)(g.origin + (long long)k * g.pitch_k + (long long)j0 * g.pitch_j + i0) * es;
    };
    if (g.pitch_k % g.pitch_j == 0) {
        const size_t rows = (size_t)(g.pitch_k / g.pitch_j);
        cudaMemcpy3DParms p = {};
        p.srcPtr = make_cudaPitchedPtr(at(src, k0), pitch, (size_t)ni * es, rows);
        p.dstPtr = make_cudaPitchedPtr(at(dst, k0), pitch, (size_t)ni * es, rows);
        p.extent = make_cudaExtent((size_t)ni * es, (size_t)nj, (size_t)(k1 - k0 + 1));
        p.kind = kind;
        return cudaMemcpy3DAsync(&p, s);
    }
    for (int k = k0; k <= k1; ++k) {
        cudaError_t e = cudaMemcpy2DAsync(at(dst, k), pitch, at(src, k), pitch, (size_t)ni * es, (size_t)nj, kind, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The host path; wait = return once the results are in host memory, else
// once the work is enqueued (the caller's stream waits for its last copy).
static pw_status_t tendencies_host(pw_handle_t h, const void* u, const void* v, const void* w, void* su, void* sv,
                                   void* sw, const float* scale, pw_stream_t stream, bool wait) {
    PW_RANGE(wait ? "pw_tendencies_host" : "pw_tendencies_host_async");
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (!u || !v || !w || !su || !sv || !sw) return fail(PW_ERR_ARG, "a field pointer is NULL");
    const pw_grid_t& g = h->grid;
    const size_t es = dtype_size(g.dtype);
    const size_t bytes = (size_t)alloc_elems_of(g) * es;
    for (auto& p : h->d_stage)
        if (!p) {
            cudaError_t e = dev_malloc(&p, bytes);
            if (e != cudaSuccess) return cuda_fail(e, "pw_tendencies_host staging allocation");
            e = cudaMemsetAsync(p, 0, bytes, reinterpret_cast<cudaStream_t>(stream));   // before the copies
            if (e != cudaSuccess) return cuda_fail(e, "pw_tendencies_host staging clear");
        }
    cudaStream_t us = reinterpret_cast<cudaStream_t>(stream);
    const void* hin[3] = {u, v, w};
    void* hout[3] = {su, sv, sw};
    // what travels: levels a..b of the inputs with their one-cell lateral
    // halo (all the scheme reads), and the interior of levels a..b of the
    // outputs
    auto copy_in = [&](int q, int a, int b, cudaStream_t s) {
        return copy_box(g, h->d_stage[q], hin[q], 0, g.nx + 2, 0, g.ny + 2, a, b, cudaMemcpyHostToDevice, s);
    };
    auto copy_out = [&](int q, int a, int b, cudaStream_t s) {
        return copy_box(g, hout[q], h->d_stage[3 + q], 1, g.nx, 1, g.ny, a, b, cudaMemcpyDeviceToHost, s);
    };

    int ox = 0;
    const char* why = "";
    bool ptrs_ok = true;
    for (auto p : h->d_stage) ptrs_ok = ptrs_ok && aligned16(p);
    const bool pipelined = h->kernel_kind != 1 && ptrs_ok && tma_layout_ok(g, &ox, &why) && g.nz >= 8;
    // Every call of either path ends by recording ev_end after its last copy
    // out.  The one-launch path runs on the caller's stream only, so it first
    // waits for the whole of the previous call (which may have run on another
    // stream); a pipelined call does the same after a one-launch call, and
    // after a pipelined call relies on the per-chunk events below.
    if (!h->ev_end) PW_CUDA(cudaEventCreateWithFlags(&h->ev_end, cudaEventDisableTiming), "pipeline event");
    if (!pipelined || h->host_prev_plain) PW_CUDA(cudaStreamWaitEvent(us, h->ev_end, 0), "pipeline wait");
    if (!pipelined) {   // one copy in, one launch, one copy out
        for (int q = 0; q < 3; ++q) PW_CUDA(copy_in(q, 1, g.nz, us), "pw_tendencies_host input copy");
        pw_status_t st = pw_tendencies(h, h->d_stage[0], h->d_stage[1], h->d_stage[2], h->d_stage[3], h->d_stage[4],
                                       h->d_stage[5], scale, stream);
        if (st != PW_OK) return st;
        for (int q = 0; q < 3; ++q) PW_CUDA(copy_out(q, 1, g.nz, us), "pw_tendencies_host output copy");
        PW_CUDA(cudaEventRecord(h->ev_end, us), "pipeline event");
        h->host_prev_plain = true;
        if (wait) PW_CUDA(cudaStreamSynchronize(us), "pw_tendencies_host synchronize");
        return PW_OK;
    }

    // Pipelined over k chunks: chunk c's input planes travel on stream 0
    // while chunk c-1 is computed on stream 1 and chunk c-2's outputs travel
    // back on stream 2 (the two copy directions and the kernels overlap).
    // Calls on one handle share the staging buffers, and a call may start
    // before the previous one has finished (the asynchronous form): chunk c's
    // input copy first waits for the previous call's kernels that read those
    // levels (chunks up to c+2), and chunk c's kernel for the previous call's
    // copy out of chunk c, so one call's inputs travel while the last one's
    // outputs come back.
    for (auto& st : h->hs)
        if (!st) PW_CUDA(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking), "pipeline stream");
    for (int c = 0; c < pw_handle_s::kMaxChunks; ++c) {
        if (!h->ev_in[c]) PW_CUDA(cudaEventCreateWithFlags(&h->ev_in[c], cudaEventDisableTiming), "pipeline event");
        if (!h->ev_comp[c]) PW_CUDA(cudaEventCreateWithFlags(&h->ev_comp[c], cudaEventDisableTiming), "pipeline event");
        if (!h->ev_out[c]) PW_CUDA(cudaEventCreateWithFlags(&h->ev_out[c], cudaEventDisableTiming), "pipeline event");
    }
    if (!h->ev_start) PW_CUDA(cudaEventCreateWithFlags(&h->ev_start, cudaEventDisableTiming), "pipeline event");
    const int C = std::min(pw_handle_s::kMaxChunks, std::max(2, g.nz / PW_HOST_CHUNK_LEVELS));
    Scales sc;
    bool scaled;
    if (scale)
        for (int q = 0; q < 6; ++q)
            if (!(scale[q] > 0.f) || !(scale[q] < 3.0e38f)) return fail(PW_ERR_ARG, "scales must be finite and > 0");
    make_scales(scale, &sc, &scaled);
    TmaConfig cfg = choose_tma(h, false);
    cfg.nseg = C;
    cfg.seg_count = 1;
    CUtensorMap maps[3];
    for (int q = 0; q < 3; ++q) {
        pw_status_t st = encode_map(h, h->d_stage[q], cfg, &maps[q]);
        if (st != PW_OK) return st;
    }
    const GridDev gd = to_dev(g);
    CoefDev cf{h->tcx, h->tcy, h->d_tz};
    PW_CUDA(cudaEventRecord(h->ev_start, us), "pipeline event");
    for (auto st : h->hs) PW_CUDA(cudaStreamWaitEvent(st, h->ev_start, 0), "pipeline wait");
    int copied = 0;   // input levels 1..copied are on their way
    for (int c = 0; c < C; ++c) {
        const int kb = 1 + (int)(((long long)c * g.nz) / C);
        const int ke = (int)(((long long)(c + 1) * g.nz) / C);
        const int need = std::min(ke + 1, g.nz);
        if (need > copied) {
            // (an event not recorded yet, as on a handle's first call, is no wait)
            PW_CUDA(cudaStreamWaitEvent(h->hs[0], h->ev_comp[std::min(c + 2, C - 1)], 0), "pipeline wait");
            for (int q = 0; q < 3; ++q)
                PW_CUDA(copy_in(q, copied + 1, need, h->hs[0]), "pw_tendencies_host input copy");
            copied = need;
        }
        PW_CUDA(cudaEventRecord(h->ev_in[c], h->hs[0]), "pipeline event");
        PW_CUDA(cudaStreamWaitEvent(h->hs[1], h->ev_in[c], 0), "pipeline wait");
        PW_CUDA(cudaStreamWaitEvent(h->hs[1], h->ev_out[c], 0), "pipeline wait");
        cfg.seg0 = c;
        cudaError_t e = launch_tend_tma(g.dtype, gd, ox, maps, h->d_stage[3], h->d_stage[4], h->d_stage[5], sc,
                                        cf, h->d_err, cfg, h->hs[1]);
        if (e != cudaSuccess) return cuda_fail(e, "TMA tendency kernel launch");
        PW_CUDA(cudaEventRecord(h->ev_comp[c], h->hs[1]), "pipeline event");
        PW_CUDA(cudaStreamWaitEvent(h->hs[2], h->ev_comp[c], 0), "pipeline wait");
        for (int q = 0; q < 3; ++q) PW_CUDA(copy_out(q, kb, ke, h->hs[2]), "pw_tendencies_host output copy");
        PW_CUDA(cudaEventRecord(h->ev_out[c], h->hs[2]), "pipeline event");
    }
    h->last_kernel = 2;
    PW_CUDA(cudaEventRecord(h->ev_end, h->hs[2]), "pipeline event");
    h->host_prev_plain = false;
    PW_CUDA(cudaStreamWaitEvent(us, h->ev_end, 0), "pipeline wait");
    if (wait) PW_CUDA(cudaStreamSynchronize(h->hs[2]), "pw_tendencies_host synchronize");
    return PW_OK;
}

pw_status_t pw_tendencies_host(pw_handle_t h, const void* u, const void* v, const void* w, void* su, void* sv,
                               void* sw, const float* scale, pw_stream_t stream) {
    return tendencies_host(h, u, v, w, su, sv, sw, scale, stream, true);
}

pw_status_t pw_tendencies_host_async(pw_handle_t h, const void* u, const void* v, const void* w, void* su, void* sv,
                                     void* sw, const float* scale, pw_stream_t stream) {
    return tendencies_host(h, u, v, w, su, sv, sw, scale, stream, false);
}

// Storage scales of a step call: the state is read and written with the same
// per-field scale (NULL = 1).
static pw_status_t step_scales(const float* scale, Scales* sc, bool* scaled) {
    *scaled = false;
    for (int q = 0; q < 3; ++q) {
        const float x = scale ? scale[q] : 1.f;
        if (!(x > 0.f) || !(x < 3.0e38f)) return fail(PW_ERR_ARG, "scales must be finite and > 0");
        sc->in[q] = x;
        sc->out[q] = 1.f / x;   // the next state is stored with the same scale
        if (x != 1.f) *scaled = true;
    }
    return PW_OK;
}

// One single-step pass src -> dst (interior levels 1..nz and the periodic
// images of the lateral halo), on the TMA k-march or the generic kernel.
static pw_status_t step_pass(pw_handle_t h, const GridDev& g, const void* const* src, void* const* dst,
                             const Scales& sc, bool scaled, const CoefDev& cf, float dt, bool use_tma, int ox,
                             const TmaConfig& c, cudaStream_t s) {
    const pw_dtype_t dtp = h->grid.dtype;
    cudaError_t e;
    if (use_tma) {
        CUtensorMap maps[3];
        for (int q = 0; q < 3; ++q) {
            pw_status_t st = encode_map(h, src[q], c, &maps[q]);
            if (st != PW_OK) return st;
        }
        e = launch_step_tma(dtp, g, ox, maps, dst[0], dst[1], dst[2], sc, cf, dt, h->d_err, c, s);
        // the single-step k-march writes the images of a one-cell halo only
        if (e == cudaSuccess && g.halo != 1) e = launch_fill_halo(dtp, g, dst, 3, h->num_sms, s);
    } else {
        e = launch_step_generic(dtp, g, src[0], src[1], src[2], dst[0], dst[1], dst[2], sc, scaled, cf, dt,
                                h->num_sms, s);
    }
    if (e != cudaSuccess) return cuda_fail(e, "step kernel launch");
    return PW_OK;
}

pw_status_t pw_step_to(pw_handle_t h, const void* u, const void* v, const void* w, void* nu, void* nv, void* nw,
                       float dt, const float* scale, pw_stream_t stream) {
    PW_RANGE("pw_step_to");
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    void* bufs[6] = {const_cast<void*>(u), const_cast<void*>(v), const_cast<void*>(w), nu, nv, nw};
    for (int a = 0; a < 6; ++a) {
        if (!bufs[a]) return fail(PW_ERR_ARG, "a field pointer is NULL");
        for (int b = 0; b < a; ++b)
            if (bufs[a] == bufs[b]) return fail(PW_ERR_ARG, "the six fields must be distinct buffers");
    }
    if (!(dt == dt) || dt > 3.0e38f || dt < -3.0e38f) return fail(PW_ERR_ARG, "dt must be finite");
    Scales sc;
    bool scaled = false;
    pw_status_t st = step_scales(scale, &sc, &scaled);
    if (st != PW_OK) return st;
    st = check_device_ptrs(h, bufs, 6);
    if (st != PW_OK) return st;
    bool use_tma = false;
    int ox = 0;
    st = march_kernel_choice(h, true, bufs, 6, &use_tma, &ox);
    if (st != PW_OK) return st;
    const GridDev g = to_dev(h->grid);
    CoefDev cf{h->tcx, h->tcy, h->d_tz};
    TmaConfig c{};
    if (use_tma) c = choose_tma(h, true);
    if (use_tma && !c.rag && h->grid.nx % c.nc)
        return fail(PW_ERR_UNSUPPORTED, "fused steps with cells=%d need nx to be a multiple of %d", c.nc, c.nc);
    st = step_pass(h, g, bufs, bufs + 3, sc, scaled, cf, dt, use_tma, ox, c, reinterpret_cast<cudaStream_t>(stream));
    if (st != PW_OK) return st;
    h->last_kernel = use_tma ? 2 : 1;
    return PW_OK;
}

pw_status_t pw_step(pw_handle_t h, void* u, void* v, void* w, void* tmp_u, void* tmp_v, void* tmp_w, float dt,
                    int32_t nsteps, const float* scale, pw_stream_t stream) {
    PW_RANGE("pw_step");
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    void* bufs[6] = {u, v, w, tmp_u, tmp_v, tmp_w};
    for (int a = 0; a < 6; ++a) {
        if (!bufs[a]) return fail(PW_ERR_ARG, "a field pointer is NULL");
        for (int b = 0; b < a; ++b)
            if (bufs[a] == bufs[b]) return fail(PW_ERR_ARG, "state and scratch buffers must be distinct");
    }
    if (nsteps < 0) return fail(PW_ERR_ARG, "nsteps must be >= 0");
    if (!(dt == dt) || dt > 3.0e38f || dt < -3.0e38f) return fail(PW_ERR_ARG, "dt must be finite");
    Scales sc;
    bool scaled = false;
    pw_status_t sst = step_scales(scale, &sc, &scaled);
    if (sst != PW_OK) return sst;
    sst = check_device_ptrs(h, bufs, 6);
    if (sst != PW_OK) return sst;
    const GridDev g = to_dev(h->grid);
    CoefDev cf{h->tcx, h->tcy, h->d_tz};
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const pw_dtype_t dtp = h->grid.dtype;
    {
        cudaError_t e = launch_fill_halo(dtp, g, bufs, 3, h->num_sms, s);
        if (e != cudaSuccess) return cuda_fail(e, "halo fill launch");
    }
    int ox = 0;
    bool use_tma = false;
    sst = march_kernel_choice(h, true, bufs, 6, &use_tma, &ox);
    if (sst != PW_OK) return sst;
    // two steps per pass: TMA path, a lateral halo >= 2, and interior rows
    // starting at least 7 elements into their padded row (the q0 box begins
    // 7 columns before the first interior column)
    const bool tb2_ok = use_tma && g.nx % 4 == 0 && g.halo >= 2 && ox >= 7;
    if (h->steps_per_pass == 2 && nsteps >= 2 && !tb2_ok)
        return fail(PW_ERR_UNSUPPORTED, "two steps per pass need the TMA path, a halo >= 2 and >= 7 columns before "
                                        "the interior in each padded row");
    // automatic (0) is one step per pass: on GB300 the two-step pass is bound
    // by instruction issue, not HBM, and runs slower per step
    const bool use_tb2 = tb2_ok && h->steps_per_pass == 2;
    TmaConfig c{};
    if (use_tma) c = choose_tma(h, true);
    if (use_tma && !c.rag && h->grid.nx % c.nc)
        return fail(PW_ERR_UNSUPPORTED, "fused steps with cells=%d need nx to be a multiple of %d", c.nc, c.nc);
    Step2Config c2{};
    if (use_tb2 && nsteps >= 2) c2 = choose_step2(h);
    int done = 0, passes = 0, kind = use_tma ? 2 : 1;
    while (done < nsteps) {
        void** src = (passes % 2 == 0) ? bufs : bufs + 3;
        void** dst = (passes % 2 == 0) ? bufs + 3 : bufs;
        if (use_tb2 && nsteps - done >= 2) {
            CUtensorMap maps[3];
            for (int q = 0; q < 3; ++q) {
                pw_status_t st = encode_map_box(h, src[q], step2_box_width(), c2.ty + 2, &maps[q]);
                if (st != PW_OK) return st;
            }
            cudaError_t e = launch_step2_tma(dtp, g, ox, maps, dst[0], dst[1], dst[2], sc, cf, dt, h->d_err, c2, s);
            done += 2;
            kind = 3;
            if (e != cudaSuccess) return cuda_fail(e, "step kernel launch");
        } else {
            pw_status_t st = step_pass(h, g, src, dst, sc, scaled, cf, dt, use_tma, ox, c, s);
            if (st != PW_OK) return st;
            done += 1;
        }
        ++passes;
    }
    h->last_kernel = kind;
    if (passes % 2 == 1) {   // the last state is in the scratch buffers: copy levels 1..nz back
        const size_t es = dtype_size(dtp);
        const pw_grid_t& gg = h->grid;
        const size_t lo = (size_t)(gg.origin + gg.pitch_k + (long long)(1 - gg.halo) * gg.pitch_j + 1 - gg.halo);
        const size_t hi = (size_t)(gg.origin + (long long)gg.nz * gg.pitch_k +
                                   (long long)(gg.ny + gg.halo) * gg.pitch_j + gg.nx + gg.halo + 1);
        for (int q = 0; q < 3; ++q)
            PW_CUDA(cudaMemcpyAsync((char*)bufs[q] + lo * es, (const char*)bufs[3 + q] + lo * es, (hi - lo) * es,
                                    cudaMemcpyDeviceToDevice, s),
                    "state copy");
    }
    return PW_OK;
}

pw_status_t pw_adjoint(pw_handle_t h, const void* u, const void* v, const void* w, const void* lsu,
                       const void* lsv, const void* lsw, void* gu, void* gv, void* gw, float alpha, int32_t flags,
                       pw_stream_t stream) {
    PW_RANGE("pw_adjoint");
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (h->grid.dtype != PW_F32) return fail(PW_ERR_UNSUPPORTED, "pw_adjoint supports FP32 fields only");
    if (!u || !v || !w || !lsu || !lsv || !lsw || !gu || !gv || !gw) return fail(PW_ERR_ARG, "a field pointer is NULL");
    if (flags & ~(PW_ADJ_ACCUMULATE | PW_ADJ_PERIODIC | PW_ADJ_ADD_LAMBDA)) return fail(PW_ERR_ARG, "unknown flag bits");
    if ((flags & PW_ADJ_ACCUMULATE) && (flags & PW_ADJ_ADD_LAMBDA))
        return fail(PW_ERR_ARG, "PW_ADJ_ACCUMULATE and PW_ADJ_ADD_LAMBDA are exclusive");
    const void* ins[6] = {u, v, w, lsu, lsv, lsw};
    const void* outs[3] = {gu, gv, gw};
    for (auto o : outs)
        for (auto i : ins)
            if (o == i) return fail(PW_ERR_ARG, "an output aliases an input");
    if (gu == gv || gu == gw || gv == gw) return fail(PW_ERR_ARG, "outputs alias each other");
    if (!(alpha == alpha) || alpha > 3.0e38f || alpha < -3.0e38f) return fail(PW_ERR_ARG, "alpha must be finite");
    {
        pw_status_t dst = check_device_ptrs(h, ins, 6);
        if (dst == PW_OK) dst = check_device_ptrs(h, outs, 3);
        if (dst != PW_OK) return dst;
    }
    CoefDev cf{h->tcx, h->tcy, h->d_tz};
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int ox = 0;
    const char* why = "";
    bool ptrs_ok = true;
    for (auto p : ins) ptrs_ok = ptrs_ok && aligned16(p);
    for (auto p : outs) ptrs_ok = ptrs_ok && aligned16(p);
    // Widths that are a multiple of 4 in periodic mode; the full array at any
    // width; and periodic ones at any width from kRagMinNx columns and
    // kShapeMinCells cells up (the ring of cells gathered by a second launch is
    // then a small part), both with the automatic shape.
    const pw_grid_t& gr = h->grid;
    const AdjMode mode = !(flags & PW_ADJ_PERIODIC) ? ADJ_OPEN : (gr.nx % 4 == 0 ? ADJ_PERIODIC : ADJ_PERIODIC_ANY);
    const bool size_ok = mode != ADJ_PERIODIC_ANY || (h->kernel_kind == 0 && gr.nx >= kRagMinNx && gr.ny >= 8 &&
                                                      (long long)gr.nx * gr.ny * gr.nz >= kShapeMinCells);
    // the full array and odd widths were the gather kernel's, which takes any height and depth
    const bool fits = mode == ADJ_PERIODIC || (gr.ny + 2LL <= 8LL * kMaxGridY && gr.nz <= 64LL * kMaxGridY);
    if (h->kernel_kind != 1 && ptrs_ok && size_ok && fits && (mode == ADJ_PERIODIC || !adj_fixed(h)) &&
        tma_layout_ok(gr, &ox, &why, mode != ADJ_PERIODIC)) {
        const GridDev g = to_dev(gr);
        if (mode == ADJ_PERIODIC) {   // the sensitivities need periodic halos too
            void* ls[3] = {const_cast<void*>(lsu), const_cast<void*>(lsv), const_cast<void*>(lsw)};
            cudaError_t e = launch_fill_halo(PW_F32, g, ls, 3, h->num_sms, s);
            if (e != cudaSuccess) return cuda_fail(e, "sensitivity halo fill");
        }
        CUtensorMap maps[6];
        const AdjConfig ac = choose_adjoint(h, mode);
        for (int q = 0; q < 6; ++q) {
            pw_status_t st = adj_map(h, q, ins[q], mode, ox, ac.lx * ac.na + 8, ac.ty + 2, &maps[q]);
            if (st != PW_OK) return st;
        }
        const float* q6[6] = {(const float*)u,   (const float*)v,   (const float*)w,
                              (const float*)lsu, (const float*)lsv, (const float*)lsw};
        float* g3[3] = {(float*)gu, (float*)gv, (float*)gw};
        cudaError_t e = launch_adjoint_tma(g, adj_geom(gr, ox, mode), mode, maps, q6, g3, alpha,
                                           (flags & PW_ADJ_ACCUMULATE) ? 1 : 0, (flags & PW_ADJ_ADD_LAMBDA) ? 1 : 0,
                                           cf, h->d_err, ac, h->num_sms, s);
        if (e != cudaSuccess) return cuda_fail(e, "adjoint kernel launch");
        h->last_kernel = 2;
        return PW_OK;
    }
    h->last_kernel = 1;
    cudaError_t e = launch_adjoint(to_dev(h->grid), (const float*)u, (const float*)v, (const float*)w,
                                   (const float*)lsu, (const float*)lsv, (const float*)lsw, (float*)gu, (float*)gv,
                                   (float*)gw, alpha, (flags & PW_ADJ_ACCUMULATE) ? 1 : 0,
                                   (flags & PW_ADJ_ADD_LAMBDA) ? 1 : 0, (flags & PW_ADJ_PERIODIC) ? 1 : 0, cf,
                                   h->num_sms, s);
    if (e != cudaSuccess) return cuda_fail(e, "adjoint kernel launch");
    return PW_OK;
}

pw_status_t pw_fill_halo_periodic(pw_handle_t h, void* f, pw_stream_t stream) {
    PW_RANGE("pw_fill_halo_periodic");
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (!f) return fail(PW_ERR_ARG, "field pointer is NULL");
    {
        const void* p = f;
        pw_status_t dst = check_device_ptrs(h, &p, 1);
        if (dst != PW_OK) return dst;
    }
    cudaError_t e = launch_fill_halo(h->grid.dtype, to_dev(h->grid), &f, 1, h->num_sms,
                                     reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "halo fill launch");
    return PW_OK;
}

pw_status_t pw_keep_interior(pw_handle_t h, const void* a, const void* b, const void* c, void* da, void* db, void* dc,
                             int64_t n, pw_stream_t stream) {
    PW_RANGE("pw_keep_interior");
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (!da || !db || !dc) return fail(PW_ERR_ARG, "a field pointer is NULL");
    if (n < alloc_elems_of(h->grid)) return fail(PW_ERR_ARG, "n is less than a field of this layout holds");
    const void* src[3] = {a, b, c};
    void* dst[3] = {da, db, dc};
    if (da == db || da == dc || db == dc) return fail(PW_ERR_ARG, "outputs alias each other");
    for (int q = 0; q < 3; ++q)
        for (int d = 0; d < 3; ++d)
            if (q != d && src[q] == dst[d]) return fail(PW_ERR_ARG, "an output aliases another field's input");
    for (int q = 0; q < 3; ++q) {
        const void* p[2] = {dst[q], src[q]};
        pw_status_t st = check_device_ptrs(h, p, src[q] ? 2 : 1);
        if (st != PW_OK) return st;
    }
    cudaError_t e = launch_keep_interior(h->grid.dtype, to_dev(h->grid), src, dst, (long long)n, h->num_sms,
                                         reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "interior copy launch");
    return PW_OK;
}

static pw_status_t ensure_scratch(pw_handle_t h) {
    if (h->d_scratch) return PW_OK;
    h->nblocks = norm_blocks(h->num_sms);
    const size_t n = 4 * (size_t)(h->nblocks + 1) + (size_t)(h->grid.nz + 2);
    cudaError_t e = dev_malloc(&h->d_scratch, n * sizeof(double));
    if (e != cudaSuccess) {
        h->d_scratch = nullptr;
        return cuda_fail(e, "validation scratch allocation");
    }
    return PW_OK;
}

pw_status_t pw_error_norms(pw_handle_t h, const void* test, float scale, const double* ref, int32_t k0, int32_t k1,
                           double* out, pw_stream_t stream) {
    PW_RANGE("pw_error_norms");
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (!test || !ref || !out) return fail(PW_ERR_ARG, "a pointer is NULL");
    if (k0 < 1 || k1 > h->grid.nz || k0 > k1) return fail(PW_ERR_ARG, "need 1 <= k0 <= k1 <= nz");
    const void* dp[2] = {test, ref};
    pw_status_t st = check_device_ptrs(h, dp, 2);
    if (st != PW_OK) return st;
    st = ensure_scratch(h);
    if (st != PW_OK) return st;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = launch_error_norms(h->grid.dtype, to_dev(h->grid), test, scale, ref, k0, k1, h->d_scratch,
                                       h->nblocks, s);
    if (e != cudaSuccess) return cuda_fail(e, "norm kernel launch");
    PW_CUDA(cudaMemcpyAsync(out, h->d_scratch + 4 * (size_t)h->nblocks, 4 * sizeof(double), cudaMemcpyDeviceToHost, s),
            "norm result copy");
    PW_CUDA(cudaStreamSynchronize(s), "norm synchronize");
    return PW_OK;
}

pw_status_t pw_weighted_dot(pw_handle_t h, const void* a, float sa, const void* b, float sb, const double* wk,
                            int32_t k0, int32_t k1, double* out, pw_stream_t stream) {
    PW_RANGE("pw_weighted_dot");
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (!a || !b || !out) return fail(PW_ERR_ARG, "a pointer is NULL");
    if (k0 < 1 || k1 > h->grid.nz || k0 > k1) return fail(PW_ERR_ARG, "need 1 <= k0 <= k1 <= nz");
    const void* dp[2] = {a, b};
    pw_status_t st = check_device_ptrs(h, dp, 2);
    if (st != PW_OK) return st;
    st = ensure_scratch(h);
    if (st != PW_OK) return st;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    double* d_wk = nullptr;
    if (wk) {
        d_wk = h->d_scratch + 4 * (size_t)(h->nblocks + 1);
        PW_CUDA(cudaMemcpyAsync(d_wk, wk, (h->grid.nz + 2) * sizeof(double), cudaMemcpyHostToDevice, s),
                "weight copy");
    }
    cudaError_t e = launch_weighted_dot(h->grid.dtype, to_dev(h->grid), a, sa, b, sb, d_wk, k0, k1, h->d_scratch,
                                        h->nblocks, s);
    if (e != cudaSuccess) return cuda_fail(e, "dot kernel launch");
    double r[4];
    PW_CUDA(cudaMemcpyAsync(r, h->d_scratch + 4 * (size_t)h->nblocks, 4 * sizeof(double), cudaMemcpyDeviceToHost, s),
            "dot result copy");
    PW_CUDA(cudaStreamSynchronize(s), "dot synchronize");
    out[0] = r[2];
    return PW_OK;
}

pw_status_t pw_sync(pw_handle_t h, pw_stream_t stream) {
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    PW_CUDA(cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(stream)), "stream synchronize");
    int flag = 0;
    PW_CUDA(cudaMemcpy(&flag, h->d_err, sizeof(int), cudaMemcpyDeviceToHost), "status word read");
    if (flag != DEV_OK) {
        cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
        PW_CUDA(cudaMemsetAsync(h->d_err, 0, sizeof(int), s), "status word clear");
        PW_CUDA(cudaStreamSynchronize(s), "status word clear");
        if (flag == DEV_OOB_STORE)
            return fail(PW_ERR_CUDA, "a store outside the field's cells was caught and skipped (debug bounds build)");
        return fail(PW_ERR_DEVICE_TIMEOUT, "a kernel gave up a bounded wait (code %d)", flag);
    }
    PW_CUDA(cudaGetLastError(), "pending CUDA error");
    return PW_OK;
}

int32_t pw_debug_layout_check(const pw_grid_t* g, int64_t offset, int32_t n, int32_t interior_only) {
    if (!g || validate_grid(g) != PW_OK || n < 1) return -1;
    return layout_cells_ok(to_dev(*g), (long long)offset, n, interior_only != 0) ? 1 : 0;
}

int32_t pw_debug_bounds_build(void) { return PW_DEBUG_BOUNDS ? 1 : 0; }

pw_status_t pw_inject_failures(int32_t kind, int32_t count) {
    if (kind < 0 || kind >= INJECT_KINDS) return fail(PW_ERR_ARG, "kind must be 0 (allocations) or 1 (tensor maps)");
    if (count < 0) return fail(PW_ERR_ARG, "count must be >= 0");
    g_inject[kind].store(count, std::memory_order_relaxed);
    return PW_OK;
}

pw_status_t pw_selftest_wait_timeout(pw_handle_t h, int64_t limit_ns, pw_stream_t stream) {
    PW_RANGE("pw_selftest_wait_timeout");
    if (!h) return fail(PW_ERR_ARG, "handle is NULL");
    if (limit_ns < 1000000 || limit_ns > 1000000000) return fail(PW_ERR_ARG, "limit_ns must be in [1e6, 1e9]");
    cudaError_t e = launch_selftest_wait((uint64_t)limit_ns, h->d_err, reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "self-test launch");
    return PW_OK;
}

const char* pw_last_error(void) { return g_err.c_str(); }

const char* pw_status_string(pw_status_t s) {
    switch (s) {
        case PW_OK: return "PW_OK";
        case PW_ERR_ARG: return "PW_ERR_ARG";
        case PW_ERR_ALIGN: return "PW_ERR_ALIGN";
        case PW_ERR_CUDA: return "PW_ERR_CUDA";
        case PW_ERR_OOM: return "PW_ERR_OOM";
        case PW_ERR_DEVICE_TIMEOUT: return "PW_ERR_DEVICE_TIMEOUT";
        case PW_ERR_UNSUPPORTED: return "PW_ERR_UNSUPPORTED";
    }
    return "PW_ERR_UNKNOWN";
}

}  // extern "C"
