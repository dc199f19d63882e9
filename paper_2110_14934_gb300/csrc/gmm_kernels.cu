// Kernels: single-camera tick, List 1 alone, the 3x3 opening of a
// bit-packed mask, mask packing and confusion counts. (The multi-camera tick
// is in gmm_pool_kernel.cu.)
//
// The tick is a stream over the mixture state: per pixel it needs about
// 24 M + 40 bytes of FP32 state (what a tick reads and changes, see
// ranked_step) and half that of FP16/BF16 state, plus 5 bytes of frame, the
// List-1 byte and 1/8 byte of mask. There is no dense contraction, so there
// is no tensor-core work; the design goal is full-line coalesced traffic
// with enough bytes in flight per SM.
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "gmm_internal.h"

using namespace gmmdev;
using gmmhost::PoolArgs;

namespace {

// ------------------------------------------------------------ single camera
// Programmatic dependent launch between consecutive ticks on a stream: a
// tick waits for the kernel before it to complete (and its writes to be
// visible) before it reads anything, then lets the next tick be scheduled,
// so the next tick's CTAs take the SMs this tick's last CTAs leave idle
// instead of waiting for a full launch. (Both are no-ops when the kernel was
// not launched as a dependent.)
__device__ __forceinline__ void dependent_launch_prologue() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A CTA ticks one run of blockDim padded pixels, one pixel per thread (n_pad
// is a multiple of 32: whole warps leave), or, kLoop, `runs` consecutive ones,
// moving the next run's state towards L2 while it ticks one. The first `early`
// CTAs, which the hardware may schedule while the kernel before this one
// drains, move their first run's state before they wait for that kernel.
template <int M, int PREC, int V, bool kLoop>
__device__ __forceinline__ void tick_body(const CamView &cv, int runs, int early) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x * (kLoop ? runs : 1) + threadIdx.x;
    if (PREC != kF16 && (int)blockIdx.x < early && p < cv.n_pad)
        prefetch_pixels<M, PREC, V>(cv, p);
    dependent_launch_prologue();
    if (!kLoop) {
        if (p >= cv.n_pad)
            return;
        const uint32_t bits = process_pixel<M, PREC, V>(cv, p);
        write_mask_words(cv, p >> 5, bits);
        return;
    }
    for (int k = 0; k < runs && p < cv.n_pad; ++k, p += blockDim.x) {
        if (k + 1 < runs && p + blockDim.x < cv.n_pad)
            prefetch_pixels<M, PREC, V>(cv, p + blockDim.x);
        const uint32_t bits = process_pixel<M, PREC, V>(cv, p);
        write_mask_words(cv, p >> 5, bits);
    }
}

// V: process_pixel's variant (the options are separate instantiations, so the
// default kernels carry none of them). The kernels wait for memory more than
// for anything else (issue slots about 60% used in FP16/BF16, less in FP32),
// so warps count: 40 per SM (48 registers, small spills) measured 63.8 us
// against 64.5 with 32 at 1920x1080, M = 5, FP32, and 43.2 against 44.4 in
// FP16/BF16 (48 warps: 47.0). Two pixels per thread spill (FP16/BF16 53.0);
// a persistent form fed by bulk copies through shared memory measured slower
// (73 against 70 at the time: a stage waits for the slowest of its warps, and
// in most tiles one of them goes to memory for a mean). Small CTAs measured
// faster than 256 threads: a CTA's slot frees as soon as its own warps finish.
// The looping form holds more values across a pixel: 64 registers in FP32 and
// for M = 5.
template <int M, int PREC, bool kLoop> struct TickBounds {
    static constexpr int kCtas = kLoop && (PREC == kF32 || M == 5) ? 4 : 5; // of 256 threads
};
template <int M, int PREC, int V, bool kLoop>
__global__ void __launch_bounds__(256, (TickBounds<M, PREC, kLoop>::kCtas))
    k_tick(const CamView cv, int runs, int early) {
    tick_body<M, PREC, V, kLoop>(cv, runs, early);
}

// Runs per CTA. Looping saves CTA turnover and hides the next run's state
// behind the current one, but leaves fewer CTAs to even out the end of the
// launch: it pays from about a dozen waves of the SMs x 1024 threads on. Measured (us; 1, 2, 4 runs): FP32 1280x720 M = 3 options 26.3,
// 27.9, 30.1; 1920x1080 M = 5 63.6, 62.7, 64.3; 2560x1440 M = 4 95.8, 92.2,
// 93.2; 3840x2160 M = 5 238, 227, 227; FP16/BF16 1920x1080 M = 3 35.5, 33.7,
// 33.8; 2560x1440 M = 4 66.7, 64.6, 63.7; 3840x2160 M = 3 133.8, 117.6, 115.7;
// M = 5 (whose looping form has 32 warps per SM against 40) 1920x1080 43.2,
// 44.4, 44.7; 3840x2160 162.8, 154.6, 150.7.
template <int M, int PREC> int tick_runs(int64_t n_pad, int sms) {
    const int64_t waves = n_pad / (sms * (int64_t)1024);
    if (waves >= 32)
        return 4;
    return waves >= (PREC != kF32 && M == 5 ? 20 : 12) ? 2 : 1;
}

template <int M, int PREC, int V>
cudaError_t launch_tick_v(const CamView &cv, int threads, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    const int sms = gmmhost::num_sms();
    const int runs = tick_runs<M, PREC>(cv.n_pad, sms);
    const int64_t px = (int64_t)threads * runs;
    // 2560 threads per SM: two waves of CTAs, two and a half of the forms that
    // keep 32 warps resident. An opening's few CTAs leave HBM idle, and so does
    // the end of a tick: with an opening after each tick FP32 1021x767 M = 4 26.7 ->
    // 25.2 us, 1280x720 M = 3 options 26.0 -> 25.1, caller-owned FP16/BF16
    // 1280x720 M = 4 22.1 -> 21.3; ticks alone FP32 1920x1080 M = 5 62.6 ->
    // 62.0. The FP16/BF16 handles' kernel loses by it (1920x1080 M = 5 43.1 ->
    // 46.5 us: more spills, and the state it would move is a smaller part of
    // its time), and does without.
    const int early = sms * 2560 / threads;
    cfg.gridDim = dim3((unsigned)((cv.n_pad + px - 1) / px));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return runs > 1 ? cudaLaunchKernelEx(&cfg, k_tick<M, PREC, V, true>, cv, runs, early)
                    : cudaLaunchKernelEx(&cfg, k_tick<M, PREC, V, false>, cv, runs, early);
}

template <int M, int PREC>
cudaError_t launch_tick_t(const CamView &cv, int threads, cudaStream_t s) {
    switch (gmmhost::view_variant(cv)) {
    case 0: return launch_tick_v<M, PREC, 0>(cv, threads, s);
    case 1: return launch_tick_v<M, PREC, 1>(cv, threads, s);
    default: return launch_tick_v<M, PREC, 2>(cv, threads, s);
    }
}

// ------------------------------------------------------------ List 1 alone
__global__ void __launch_bounds__(256) k_fuse(const uint32_t *fg_rgb, const uint32_t *fg_d,
                                              uint8_t *fusion, uint32_t *mask, int H, int W,
                                              int wpr) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n_pad = (int64_t)H * wpr * 32;
    if (p >= n_pad)
        return;
    const int64_t wi = p >> 5;
    const int64_t row = wi / wpr;
    const int x = (int)(p - row * wpr * 32);
    const int lane = (int)(p & 31);
    uint32_t F = 0u;
    if (x < W) {
        const int fc = (int)((fg_rgb[wi] >> lane) & 1u);
        const int fd = (int)((fg_d[wi] >> lane) & 1u);
        const int64_t q = row * W + x;
        const uint32_t fb = fuse_list1(fc, fd, fusion[q]);
        fusion[q] = (uint8_t)fb;
        F = fb & 1u;
    }
    const uint32_t word = __ballot_sync(0xffffffffu, F);
    if (lane == 0)
        mask[wi] = word;
}

// ------------------------------------------------------------ 3x3 opening
// A CTA of 32 x 8 threads produces an 8-row x 32-word tile. It stages the
// input tile with a 2-row and 2-word halo in shared memory, erodes (AND of
// the 3x3 neighbourhood, outside = 0) into a 1-row/1-word halo, then dilates
// (OR) into the output. Bit i of a word is pixel 32*word + i, so the left
// neighbour of bit i is bit i-1 (x << 1) and bit 0 takes bit 31 of the word
// on the left.
constexpr int kMR = 8, kMW = 32;

__device__ __forceinline__ uint32_t row_valid_bits(int w, int wpr, int W) {
    if (w < 0 || w >= wpr)
        return 0u;
    const int rem = W - 32 * w;
    return rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u);
}

__global__ void __launch_bounds__(kMR * kMW) k_morph_open3(const uint32_t *in, uint32_t *out,
                                                          int H, int W, int wpr) {
    __shared__ uint32_t s_in[kMR + 4][kMW + 4];  // rows r0-2.., words w0-2..
    __shared__ uint32_t s_h[kMR + 4][kMW + 2];   // horizontal erosion, words w0-1..
    __shared__ uint32_t s_e[kMR + 2][kMW + 2];   // erosion, rows r0-1.., words w0-1..
    __shared__ uint32_t s_hd[kMR + 2][kMW];      // horizontal dilation, words w0..
    dependent_launch_prologue(); // the mask it reads is complete; the next tick may be scheduled
    const int r0 = blockIdx.y * kMR, w0 = blockIdx.x * kMW;
    const int tid = threadIdx.y * kMW + threadIdx.x, nt = kMR * kMW;

    for (int i = tid; i < (kMR + 4) * (kMW + 4); i += nt) {
        const int rr = i / (kMW + 4), ww = i % (kMW + 4);
        const int r = r0 - 2 + rr, w = w0 - 2 + ww;
        uint32_t v = 0u;
        if (r >= 0 && r < H && w >= 0 && w < wpr)
            v = in[(int64_t)r * wpr + w] & row_valid_bits(w, wpr, W);
        s_in[rr][ww] = v;
    }
    __syncthreads();
    for (int i = tid; i < (kMR + 4) * (kMW + 2); i += nt) {
        const int rr = i / (kMW + 2), ww = i % (kMW + 2);
        const uint32_t m = s_in[rr][ww + 1], l = s_in[rr][ww], r = s_in[rr][ww + 2];
        s_h[rr][ww] = m & ((m << 1) | (l >> 31)) & ((m >> 1) | (r << 31));
    }
    __syncthreads();
    for (int i = tid; i < (kMR + 2) * (kMW + 2); i += nt) {
        const int rr = i / (kMW + 2), ww = i % (kMW + 2);
        const int r = r0 - 1 + rr, w = w0 - 1 + ww;
        uint32_t e = s_h[rr][ww] & s_h[rr + 1][ww] & s_h[rr + 2][ww];
        if (r < 0 || r >= H)
            e = 0u;
        s_e[rr][ww] = e & row_valid_bits(w, wpr, W);
    }
    __syncthreads();
    for (int i = tid; i < (kMR + 2) * kMW; i += nt) {
        const int rr = i / kMW, ww = i % kMW;
        const uint32_t m = s_e[rr][ww + 1], l = s_e[rr][ww], r = s_e[rr][ww + 2];
        s_hd[rr][ww] = m | (m << 1) | (l >> 31) | (m >> 1) | (r << 31);
    }
    __syncthreads();
    const int r = r0 + threadIdx.y, w = w0 + threadIdx.x;
    if (r < H && w < wpr) {
        const int rr = threadIdx.y + 1;
        const uint32_t o = s_hd[rr - 1][threadIdx.x] | s_hd[rr][threadIdx.x] | s_hd[rr + 1][threadIdx.x];
        out[(int64_t)r * wpr + w] = o & row_valid_bits(w, wpr, W);
    }
}

// ------------------------------------------------------------ mask metrics
// Byte mask (H*W, non-zero = 1) to the bit-packed layout: one thread per
// padded pixel, one ballot per word.
__global__ void __launch_bounds__(256) k_pack(const uint8_t *in, uint32_t *out, int H, int W,
                                              int wpr) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= (int64_t)H * wpr * 32)
        return;
    const int64_t row = (p >> 5) / wpr;
    const int x = (int)(p - row * wpr * 32);
    const uint32_t b = (x < W && in[row * W + x] != 0) ? 1u : 0u;
    const uint32_t word = __ballot_sync(0xffffffffu, b);
    if ((p & 31) == 0)
        out[p >> 5] = word;
}

// Confusion counts of a predicted mask against a truth mask (both
// bit-packed, bits beyond W ignored): out = {TP, FP, FN, TN}, accumulated.
__global__ void __launch_bounds__(256) k_confusion(const uint32_t *pred, const uint32_t *truth,
                                                   int H, int W, int wpr,
                                                   unsigned long long *out) {
    unsigned long long c[4] = {0, 0, 0, 0}; // TP, FP, FN, TN
    const int64_t n_words = (int64_t)H * wpr;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_words;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int col = (int)(i % wpr);
        const int rem = W - 32 * col;
        const uint32_t valid = rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u);
        const uint32_t p = pred[i], t = truth[i];
        c[0] += __popc(p & t & valid);
        c[1] += __popc(p & ~t & valid);
        c[2] += __popc(~p & t & valid);
        c[3] += __popc(~p & ~t & valid);
    }
    __shared__ unsigned long long s[4][8]; // blockDim.x = 256: 8 warps
#pragma unroll
    for (int k = 0; k < 4; ++k)
        for (int off = 16; off > 0; off >>= 1)
            c[k] += __shfl_xor_sync(0xffffffffu, c[k], off);
    if ((threadIdx.x & 31) == 0)
        for (int k = 0; k < 4; ++k)
            s[k][threadIdx.x >> 5] = c[k];
    __syncthreads();
    if (threadIdx.x < 4) {
        unsigned long long v = 0;
        for (int w = 0; w < 8; ++w)
            v += s[threadIdx.x][w];
        atomicAdd(&out[threadIdx.x], v);
    }
}

} // namespace

namespace gmmhost {

cudaError_t launch_tick(const CamView &cv, int threads, cudaStream_t s) {
    if (cv.n_pad == 0)
        return cudaSuccess;
    if (threads != 32 && threads != 64 && threads != 128 && threads != 256)
        return cudaErrorInvalidValue;
    if (cv.prec == kF32) {
        switch (cv.M) {
        case 3: return launch_tick_t<3, kF32>(cv, threads, s);
        case 4: return launch_tick_t<4, kF32>(cv, threads, s);
        case 5: return launch_tick_t<5, kF32>(cv, threads, s);
        }
    } else if (cv.prec == kF16) {
        switch (cv.M) {
        case 3: return launch_tick_t<3, kF16>(cv, threads, s);
        case 4: return launch_tick_t<4, kF16>(cv, threads, s);
        case 5: return launch_tick_t<5, kF16>(cv, threads, s);
        }
    } else {
        switch (cv.M) {
        case 3: return launch_tick_t<3, kF16Caller>(cv, threads, s);
        case 4: return launch_tick_t<4, kF16Caller>(cv, threads, s);
        case 5: return launch_tick_t<5, kF16Caller>(cv, threads, s);
        }
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_fuse(const uint32_t *fg_rgb, const uint32_t *fg_d, uint8_t *fusion,
                        uint32_t *mask, int H, int W, cudaStream_t s) {
    const int wpr = (W + 31) / 32;
    const int64_t n_pad = (int64_t)H * wpr * 32;
    if (n_pad == 0)
        return cudaSuccess;
    k_fuse<<<(unsigned)((n_pad + 255) / 256), 256, 0, s>>>(fg_rgb, fg_d, fusion, mask, H, W, wpr);
    return cudaGetLastError();
}

cudaError_t launch_morph_open3(const uint32_t *in, uint32_t *out, int H, int W, cudaStream_t s) {
    const int wpr = (W + 31) / 32;
    // a programmatic dependent of the kernel before it, like the ticks
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)((wpr + kMW - 1) / kMW), (unsigned)((H + kMR - 1) / kMR));
    cfg.blockDim = dim3(kMW, kMR);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_morph_open3, in, out, H, W, wpr);
}

cudaError_t launch_pack(const uint8_t *in, uint32_t *out, int H, int W, cudaStream_t s) {
    const int wpr = (W + 31) / 32;
    const int64_t n = (int64_t)H * wpr * 32;
    if (n == 0)
        return cudaSuccess;
    k_pack<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(in, out, H, W, wpr);
    return cudaGetLastError();
}

cudaError_t launch_confusion(const uint32_t *pred, const uint32_t *truth, int H, int W,
                             unsigned long long *out, cudaStream_t s) {
    const int wpr = (W + 31) / 32;
    const int64_t n_words = (int64_t)H * wpr;
    cudaError_t e = cudaMemsetAsync(out, 0, 4 * sizeof(unsigned long long), s);
    if (e != cudaSuccess || n_words == 0)
        return e;
    int64_t blocks = (n_words + 255) / 256;
    const int64_t cap = (int64_t)num_sms() * 8;
    if (blocks > cap)
        blocks = cap;
    k_confusion<<<(unsigned)blocks, 256, 0, s>>>(pred, truth, H, W, wpr, out);
    return cudaGetLastError();
}

// SMs of the current device (asked for once per device).
int num_sms() {
    static std::atomic<int> known[64];
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess)
        return 1;
    std::atomic<int> *slot = dev >= 0 && dev < 64 ? &known[dev] : nullptr;
    if (slot && (n = slot->load(std::memory_order_relaxed)) > 0)
        return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    if (slot)
        slot->store(n, std::memory_order_relaxed);
    return n;
}

} // namespace gmmhost
