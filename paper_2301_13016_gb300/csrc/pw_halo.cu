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
// blockIdx.y = field: one launch for the fields of a state (three launches of
// one field each cost 3 x 2.2 us on an idle GPU at 512^2 x 64, one 3.1 us).
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
// = field.  One pass of 8 bytes an element (4 in place) instead of a mask, a
// select and a masked fill per field: those took 0.19 ms of the 512^2 x 64
// rollout's backward, this 0.07.
struct KeepFields {
    const void* src[3];
    void* dst[3];
};
template <typename E>
__global__ void keep_interior_kernel(const GridDev g, const KeepFields fs, const long long n) {
    const E* const src = reinterpret_cast<const E*>(fs.src[blockIdx.y]);
    E* const dst = reinterpret_cast<E*>(fs.dst[blockIdx.y]);
    const bool in_place = static_cast<const void*>(src) == static_cast<const void*>(dst);
    for (long long e0 = blockIdx.x * (long long)blockDim.x; e0 < n; e0 += (long long)gridDim.x * blockDim.x) {
        const long long e = e0 + threadIdx.x;
        if (e >= n) break;
        const long long rel = e - g.origin;
        bool in = rel > 0;
        if (in) {
            long long k, r, j;
            if (n < (1ll << 32)) {
                const unsigned q = (unsigned)rel, pk = (unsigned)g.pk, pj = (unsigned)g.pj;
                k = q / pk;
                r = q - (unsigned)k * pk;
                j = (unsigned)r / pj;
            } else {
                k = rel / g.pk;
                r = rel - k * g.pk;
                j = r / g.pj;
            }
            const long long i = r - j * g.pj;
            in = k >= 1 && k <= g.nz && j >= 1 && j <= g.ny && i >= 1 && i <= g.nx;
        }
        if (!in)
            dst[e] = E(0);
        else if (!in_place)
            dst[e] = src ? src[e] : E(0);
    }
}

cudaError_t launch_keep_interior(pw_dtype_t dt, const GridDev& g, const void* const* src, void* const* dst, long long n,
                                 int num_sms, cudaStream_t s) {
    KeepFields fs{};
    for (int q = 0; q < 3; ++q) {
        fs.src[q] = src[q];
        fs.dst[q] = dst[q];
    }
    const int threads = 256;
    const dim3 grid((unsigned)std::max(1LL, std::min<long long>((n + threads - 1) / threads, (long long)num_sms * 16)), 3);
    if (dtype_size(dt) == 4)
        keep_interior_kernel<uint32_t><<<grid, threads, 0, s>>>(g, fs, n);
    else
        keep_interior_kernel<uint16_t><<<grid, threads, 0, s>>>(g, fs, n);
    return cudaGetLastError();
}

}  // namespace pw
