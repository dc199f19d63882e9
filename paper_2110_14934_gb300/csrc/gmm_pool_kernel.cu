// Multi-camera tick: one launch advances every camera of a pool that has a
// submitted frame (up to kPoolViews cameras per launch), with the per-pixel
// arithmetic of the single-camera kernel (gmm_device.cuh), in a persistent
// form (CTAs loop over tiles) or a flat one (one chunk per warp).
#include <cuda_runtime.h>
#include <stdint.h>

#include "gmm_internal.h"

using namespace gmmdev;
using gmmhost::PoolArgs;

namespace {

// ------------------------------------------------------------ kernel
// CTAs take tiles of the implicit worklist (PoolArgs) from an atomic counter;
// the camera of a tile is found by binary search over tile_begin. The
// launch's PoolArgs are kernel parameters (24 KB of the 32 KB there may be):
// the views are read from the constant bank where they are used, hold no
// registers across a pixel's arithmetic, and reach the device with the launch
// itself. (Copied into constant memory before each launch, which also had to
// wait for the last user of that memory, they cost a tick 9 to 12 us: 24
// FP16/BF16 cameras of odd sizes 311 against 301 us, 4 cameras 52 against 44.)
// Ticks are programmatic dependents, like the single-camera ones.
__device__ __forceinline__ void dependent_launch_prologue() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// kPF: the state of a warp's next 32 pixels of the tile moves towards L2 while
// it works on the current ones (64 FP32 cameras 1361 -> 1279 us, 24 FP16/BF16
// ones of odd sizes 340 -> 330; two steps ahead 1338 and 337, with the List-1
// bytes 1309 and 333; with the frame values a step ahead in registers, which
// spill, 1315 and 331).
template <int M, int PREC, int V, bool kPF>
__device__ __forceinline__ void pool_tile(const CamView &cv, int64_t p0, int64_t p1) {
    for (int64_t p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
        // p1 - p0 is a multiple of 32 and blockDim too: warps stay whole.
        if (kPF && p + blockDim.x < p1)
            prefetch_pixels<M, PREC, V>(cv, p + blockDim.x);
        const uint32_t bits = process_pixel<M, PREC, V>(cv, p);
        write_mask_words(cv, p >> 5, bits);
    }
}

template <int M, int PREC, bool kAll, bool kPF>
__device__ __forceinline__ void pool_tile_v(const CamView &cv, int64_t p0, int64_t p1) {
    if (!kAll) {
        pool_tile<M, PREC, 0, kPF>(cv, p0, p1);
        return;
    }
    switch (gmmhost::view_variant(cv)) {
    case 0: pool_tile<M, PREC, 0, kPF>(cv, p0, p1); break;
    case 1: pool_tile<M, PREC, 1, kPF>(cv, p0, p1); break;
    default: pool_tile<M, PREC, 2, kPF>(cv, p0, p1); break;
    }
}

// Camera of tile t: the last job with tile_begin <= t (0 past the end).
__device__ __forceinline__ int tile_job(const PoolArgs &a, int64_t t) {
    int lo = 0, hi = a.n_jobs - 1;
    if (t < a.n_tiles) {
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.tile_begin[mid] <= t)
                lo = mid;
            else
                hi = mid - 1;
        }
    }
    return lo;
}

// kAll: tiles may come from cameras that use the options or the
// augmentation alternative (launched only when such a camera is in the tick).
// Registers: 64 (32 resident warps per SM; FP16/BF16 at 48 and 40 warps spills
// and measures 331 us against 322 on 24 cameras of odd sizes), the FP32
// instance that also handles the options 80. Thread 0 takes a tile from the
// counter and publishes it between two barriers. (Taking the next tile at the
// start of the current one and prefetching its head measured 913 us against
// 842 on 64 FP16/BF16 cameras, each at its best launch shape, now that a tile
// prefetches within itself.)
template <int PREC, bool kAll, bool kPF>
__global__ void __launch_bounds__(256, PREC == 0 && kAll ? 3 : 4)
    k_pool_tick(const __grid_constant__ PoolArgs a) {
    dependent_launch_prologue();
    __shared__ int64_t s_tile;
    __shared__ int s_job;
    if (blockIdx.x == 0) // the next tick's counters (their last users have finished)
        for (int i = threadIdx.x; i < a.n_reset; i += blockDim.x)
            a.reset[i] = 0;
    for (;;) {
        if (threadIdx.x == 0) {
            s_tile = atomicAdd(a.counter, 1);
            s_job = tile_job(a, s_tile);
        }
        __syncthreads();
        const int64_t t = s_tile;
        const int job = s_job;
        __syncthreads();
        if (t >= a.n_tiles)
            return;
        const CamView &cv = a.views[job];
        const int64_t p0 = (t - a.tile_begin[job]) * a.tile_pixels;
        const int64_t p1 = min(p0 + (int64_t)a.tile_pixels, cv.n_pad);
        switch (cv.M) {
        case 3: pool_tile_v<3, PREC, kAll, kPF>(cv, p0, p1); break;
        case 4: pool_tile_v<4, PREC, kAll, kPF>(cv, p0, p1); break;
        default: pool_tile_v<5, PREC, kAll, kPF>(cv, p0, p1); break;
        }
    }
}

// Non-persistent form: every warp takes one chunk of the launch's implicit
// chunk list (tile_begin counts chunks here: 32 pixels in FP32, one per lane;
// 64 in FP16/BF16, two per lane with the second pixel's loads overlapping
// the first one's arithmetic) and finds its camera by binary search. No counter and no loop: a CTA's slot frees as soon
// as its own warps finish, and no registers carry a loop across pixels.
template <int M, int PREC, int V>
__device__ __forceinline__ void flat_chunk(const CamView &cv, int64_t base) {
    const int lane = threadIdx.x & 31;
    if constexpr (PREC == 0) { // n_pad is a multiple of 32: the chunk is whole
        const int64_t p = base + lane;
        write_mask_words(cv, p >> 5, process_pixel<M, PREC, V>(cv, p));
    } else {
        uint32_t bits[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int64_t p = base + 32 * u + lane;
            bits[u] = p < cv.n_pad ? process_pixel<M, PREC, V>(cv, p) : 0u;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (base + 32 * u < cv.n_pad)
                write_mask_words(cv, (base >> 5) + u, bits[u]);
    }
}

template <int M, int PREC, bool kAll>
__device__ __forceinline__ void flat_chunk_v(const CamView &cv, int64_t base) {
    if (!kAll) {
        flat_chunk<M, PREC, 0>(cv, base);
        return;
    }
    switch (gmmhost::view_variant(cv)) {
    case 0: flat_chunk<M, PREC, 0>(cv, base); break;
    case 1: flat_chunk<M, PREC, 1>(cv, base); break;
    default: flat_chunk<M, PREC, 2>(cv, base); break;
    }
}

// MM: every camera of the launch has M = MM (the host groups the flat
// form's launches by M, so each runs a body specialised to its M), or 0
// (any M, switched per warp). FP32: no residency hint; FP16/BF16: 64
// registers, as in the other kernels.
template <int PREC, bool kAll, int MM>
__global__ void __launch_bounds__(256, PREC == 0 ? 1 : 4)
    k_pool_flat(const __grid_constant__ PoolArgs a) {
    dependent_launch_prologue();
    if (blockIdx.x == 0) // the next tick's counters, as the persistent form does
        for (int i = threadIdx.x; i < a.n_reset; i += blockDim.x)
            a.reset[i] = 0;
    const int64_t c = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (c >= a.n_tiles)
        return;
    int lo = 0, hi = a.n_jobs - 1;
    while (lo < hi) { // last job with tile_begin <= c (uniform across the warp)
        const int mid = (lo + hi + 1) >> 1;
        if (a.tile_begin[mid] <= c)
            lo = mid;
        else
            hi = mid - 1;
    }
    const CamView &cv = a.views[lo];
    const int64_t base = (c - a.tile_begin[lo]) * a.tile_pixels;
    if (MM != 0) {
        flat_chunk_v<MM != 0 ? MM : 3, PREC, kAll>(cv, base);
        return;
    }
    switch (cv.M) {
    case 3: flat_chunk_v<3, PREC, kAll>(cv, base); break;
    case 4: flat_chunk_v<4, PREC, kAll>(cv, base); break;
    default: flat_chunk_v<5, PREC, kAll>(cv, base); break;
    }
}

template <int PREC, bool kAll>
auto flat_kernel(int m) {
    switch (m) {
    case 3: return k_pool_flat<PREC, kAll, 3>;
    case 4: return k_pool_flat<PREC, kAll, 4>;
    case 5: return k_pool_flat<PREC, kAll, 5>;
    default: return k_pool_flat<PREC, kAll, 0>;
    }
}

} // namespace

namespace gmmhost {

cudaError_t launch_pool_tick_impl(const PoolArgs &args, int threads, int blocks, int prec,
                                  bool all_variants, bool flat, int m, bool prefetch,
                                  cudaStream_t s) {
    void (*kernel)(PoolArgs);
    if (flat && prec == 0)
        kernel = all_variants ? flat_kernel<0, true>(m) : flat_kernel<0, false>(m);
    else if (flat)
        kernel = all_variants ? flat_kernel<1, true>(m) : flat_kernel<1, false>(m);
    else if (prec == 0)
        kernel = all_variants ? k_pool_tick<0, true, true> : k_pool_tick<0, false, true>;
    else if (all_variants)
        kernel = k_pool_tick<1, true, false>;
    else
        kernel = prefetch ? k_pool_tick<1, false, true> : k_pool_tick<1, false, false>;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args);
}

int pool_max_ctas_per_sm(int prec, int threads) {
    int n = 0;
    cudaError_t e = prec == 0
        ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_pool_tick<0, false, true>, threads, 0)
        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_pool_tick<1, false, true>, threads, 0);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n < 1 ? 1 : n;
}

} // namespace gmmhost
