// Per-pixel device code shared by the single-camera tick kernel and the
// multi-camera persistent kernel: state loads/stores for both storage
// precisions, one mixture step (match, update or replace, re-rank,
// background test), List-1 fusion, and the bit-packed mask write.
//
// State layout in device memory (one camera). Pixels are numbered in padded
// row-major order p = row * w_pad + x (rows padded to a multiple of 32 pixels,
// so the 32 pixels of a warp map to one mask word) and grouped into tiles of
// kTile = 256 consecutive pixels. Each tile stores the 8M values of its
// pixels contiguously (8M * kTile elements), component-major (i the rank;
// fields w_c, mu_r, mu_g, mu_b, v_c, w_d, mu_d, v_d):
//   FP32: one plane per field, element (8 i + field) * kTile + t for tile
//         pixel t: a warp reads 32 consecutive floats of a plane, one fully
//         used 128-byte line;
//   FP16/BF16: two groups of four 2-byte slots per component and pixel,
//         group 0 = {w_c, w_d, mu_r, mu_g}, group 1 = {mu_b, v_c, mu_d, v_d},
//         element ((2 i + group) * kTile + t) * 4 + slot: one 8-byte access
//         moves a group (a warp: 256 contiguous bytes), and each 4-byte half
//         holds two values of one type, converted by one packed instruction.
// The offsets of a pixel's values are compile-time constants from one base
// address, and a tile's whole state is one contiguous block that a single
// bulk copy moves. The List-1 byte of a pixel lives in a separate byte array
// indexed by p (n_tiles * kTile bytes).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace gmmdev {

constexpr int kFields = 8;
constexpr int kTile = 256; // pixels per state tile
enum { F_WC = 0, F_MUR, F_MUG, F_MUB, F_VC, F_WD, F_MUD, F_VD };
constexpr uint32_t kDepthStarted = 16u;
constexpr int kStageInputs = 1;   // CamView.flags: frame bytes staged with the state
constexpr int kModeAugmented = 2; // CamView.flags: one 4-channel mixture (R, G, B, s*depth)
constexpr int kStochasticWeights = 4; // CamView.flags: BF16 weights stored with stochastic rounding
constexpr uint32_t kRhoEta = 1u;        // StreamPrm.flags: rho = alpha * eta(x | mu, sigma)
constexpr uint32_t kVarPerChannel = 2u; // StreamPrm.flags: v is the per-channel variance

// Group and slot of a field in the FP16/BF16 layout.
__host__ __device__ constexpr int h16_group(int f) {
    return (f == F_MUB || f == F_VC || f == F_MUD || f == F_VD) ? 1 : 0;
}
__host__ __device__ constexpr int h16_slot(int f) {
    return (f == F_WC || f == F_MUB) ? 0 : (f == F_WD || f == F_VC) ? 1
                                     : (f == F_MUR || f == F_MUD) ? 2 : 3;
}
// Element index, within its tile, of field f of component i at tile pixel t.
template <int PREC> __host__ __device__ constexpr int tile_elem(int i, int f, int t) {
    return PREC == 0 ? (kFields * i + f) * kTile + t
                     : ((2 * i + h16_group(f)) * kTile + t) * 4 + h16_slot(f);
}

struct StreamPrm {
    float alpha, oma, k2, T, init_var, init_w, v_min;
    uint32_t flags; // kRhoEta | kVarPerChannel
};

// Learning rate of the matched component: alpha, or with kRhoEta
// alpha * N(x; mu, sigma^2 I) (Stauffer-Grimson's rho) from the distance d2
// and variance v before the update, sigma^2 = v (kVarPerChannel) or v / D,
// capped at 1. Returns rho and sets orho = 1 - rho (oma exactly by default).
template <int D>
__device__ __forceinline__ float match_rate(const StreamPrm &p, float d2, float v, float &orho) {
    if (!(p.flags & kRhoEta)) {
        orho = p.oma;
        return p.alpha;
    }
    const float s2 = (p.flags & kVarPerChannel) ? v : v / (float)D;
    const float base = 6.28318530717958647692f * s2;
    float norm;
    if (D == 1)
        norm = 1.0f / sqrtf(base);
    else if (D == 3)
        norm = 1.0f / (base * sqrtf(base));
    else if (D == 4)
        norm = 1.0f / (base * base);
    else
        norm = powf(base, -0.5f * (float)D);
    const float rho = fminf(p.alpha * norm * expf(-d2 / (2.0f * s2)), 1.0f);
    orho = 1.0f - rho;
    return rho;
}

// Squared distance that feeds the variance: per channel with kVarPerChannel.
template <int D>
__device__ __forceinline__ float var_sample(const StreamPrm &p, float d2) {
    return (p.flags & kVarPerChannel) ? d2 / (float)D : d2;
}

// Everything one tick of one camera needs; passed by value to the
// single-camera kernel, read from constant memory by the pooled kernel.
struct CamView {
    void *planes;          // n_tiles tiles of M*8 planes of kTile elements
    uint8_t *fusion;       // n_tiles*kTile List-1 bytes, indexed by padded pixel
    const uint8_t *rgb;    // H*W*3, interleaved
    const uint16_t *depth; // H*W, millimetres, 0 = invalid
    uint32_t *mask;        // H*wpr words: fused foreground
    uint32_t *fg_rgb;      // optional colour foreground words (may be null)
    uint32_t *fg_d;        // optional depth foreground words (may be null)
    int64_t n_tiles;       // state tiles: ceil(n_pad / kTile)
    int64_t n_pad;         // H*w_pad (< 2^30)
    int H, W, w_pad, wpr;  // wpr = words per mask row = w_pad / 32
    int M, prec, first, flags; // flags: kStageInputs, kModeAugmented, kStochasticWeights
    uint32_t wpr_mul, wpr_shift; // n / wpr == umulhi(n, wpr_mul) >> wpr_shift (wpr > 1)
    float depth_scale;           // augmented mode: depth (mm) to the colour byte range
    uint32_t tick;               // ticks the model has taken (seeds stochastic rounding)
    StreamPrm pc, pd;
};

// Row of mask word n (n < 2^31): division by the words-per-row constant as a
// multiply-high and shift. With l = ceil(log2 d) and m = ceil(2^(31+l) / d),
// m < 2^32 and floor(n m / 2^(31+l)) = floor(n / d) for every n < 2^31
// (Granlund and Montgomery, "Division by invariant integers using
// multiplication", PLDI 1994).
__device__ __forceinline__ uint32_t div_wpr(uint32_t n, const CamView &cv) {
    return cv.wpr == 1 ? n : (__umulhi(n, cv.wpr_mul) >> cv.wpr_shift);
}

// ------------------------------------------------------------ storage types
// FP16/BF16 state: means and variances in float16, weights in bfloat16
// (weights need range near zero more than mantissa), converted in pairs.
// bfloat16 -> float is exact (the bits move up); float -> bfloat16 rounds to
// nearest even; float -> float16 rounds to nearest even and saturates at the
// largest finite value instead of becoming infinite.
__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }
__device__ __forceinline__ float2 f16x2_unpack(uint32_t u) {
    return __half22float2(*reinterpret_cast<const __half2 *>(&u));
}
__device__ __forceinline__ uint32_t bf16x2_pack(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint32_t f16x2_pack_sat(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Stochastic rounding of non-negative floats to bfloat16 (the weights):
// adding 16 uniform random bits below the kept ones and truncating rounds up
// with probability equal to the dropped fraction, so the stored weight is
// unbiased. The bits come from a counter-based hash of (tick, pixel, value):
// MurmurHash3's 32-bit finaliser (Appleby), applied twice.
__device__ __forceinline__ uint32_t fmix32(uint32_t h) {
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}
__device__ __forceinline__ uint32_t sr_bits(uint32_t tick, uint32_t p, uint32_t k) {
    return fmix32(fmix32(tick * 0x9e3779b9u + p) ^ (k * 0x27d4eb2fu));
}
__device__ __forceinline__ uint32_t bf16x2_pack_sr(float lo, float hi, uint32_t r) {
    const uint32_t l = (__float_as_uint(lo) + (r & 0xffffu)) >> 16;
    const uint32_t h = (__float_as_uint(hi) + (r >> 16)) & 0xffff0000u;
    return h | l;
}

// The eight values of one component at one pixel.
struct Fields {
    float wc, mur, mug, mub, vc, wd, mud, vd;
};

// Store component i (FP16/BF16 state) of the pixel in column t of the tile
// that starts at element tb. sr: nonzero = 32 random bits for the stochastic
// rounding of the two weights (kSR builds only).
template <bool kSR>
__device__ __forceinline__ void store_fields_f16(void *pl, int64_t tb, uint32_t t, int i,
                                                 const Fields &f, uint32_t sr) {
    uint2 *g = static_cast<uint2 *>(pl) + (tb >> 2) + t + 2 * i * kTile;
    const uint32_t w = (kSR && sr) ? bf16x2_pack_sr(f.wc, f.wd, sr) : bf16x2_pack(f.wc, f.wd);
    g[0] = make_uint2(w, f16x2_pack_sat(f.mur, f.mug));
    g[kTile] = make_uint2(f16x2_pack_sat(f.mub, f.vc), f16x2_pack_sat(f.mud, f.vd));
}

// ------------------------------------------------------------ mixture step
// Sort key of a component: the bits of w / sqrt(v) (a positive float, so its
// bits order like its value) with the low three bits replaced by 7 - the
// component's stored rank i. Comparing keys as unsigned integers orders by
// w / sigma and, between values that agree to 2^-20 relative (the same value
// included), puts the lower stored rank first: a total order, under which the
// network's result is the stable sort. (Two values that close lie well inside
// the 1e-5 margin at which a decision counts as near its threshold.)
__device__ __forceinline__ uint32_t rank_key(float w, float v, int i) {
    return (__float_as_uint(w * rsqrtf(v)) & ~7u) | (7u - (uint32_t)i);
}

template <int D> struct Comp {
    uint32_t key; // rank_key of the component
    float w, v;
    float mu[D];
};

template <int D>
__device__ __forceinline__ void comp_swap_if(Comp<D> &a, Comp<D> &b) {
    // a sits before b: the larger key goes first
    const bool sw = b.key > a.key;
    Comp<D> lo = sw ? b : a;
    Comp<D> hi = sw ? a : b;
    a = lo;
    b = hi;
}

// Optimal compare-exchange networks for 3, 4 and 5 elements.
template <int M, int D> __device__ __forceinline__ void rank_sort(Comp<D> (&c)[M]);
template <> __device__ __forceinline__ void rank_sort<3, 3>(Comp<3> (&c)[3]) {
    comp_swap_if(c[0], c[1]); comp_swap_if(c[0], c[2]); comp_swap_if(c[1], c[2]);
}
template <> __device__ __forceinline__ void rank_sort<3, 1>(Comp<1> (&c)[3]) {
    comp_swap_if(c[0], c[1]); comp_swap_if(c[0], c[2]); comp_swap_if(c[1], c[2]);
}
template <> __device__ __forceinline__ void rank_sort<3, 4>(Comp<4> (&c)[3]) {
    comp_swap_if(c[0], c[1]); comp_swap_if(c[0], c[2]); comp_swap_if(c[1], c[2]);
}
template <int D> __device__ __forceinline__ void net4(Comp<D> (&c)[4]) {
    comp_swap_if(c[0], c[1]); comp_swap_if(c[2], c[3]); comp_swap_if(c[0], c[2]);
    comp_swap_if(c[1], c[3]); comp_swap_if(c[1], c[2]);
}
template <> __device__ __forceinline__ void rank_sort<4, 3>(Comp<3> (&c)[4]) { net4(c); }
template <> __device__ __forceinline__ void rank_sort<4, 1>(Comp<1> (&c)[4]) { net4(c); }
template <> __device__ __forceinline__ void rank_sort<4, 4>(Comp<4> (&c)[4]) { net4(c); }
template <int D> __device__ __forceinline__ void net5(Comp<D> (&c)[5]) {
    comp_swap_if(c[0], c[1]); comp_swap_if(c[3], c[4]); comp_swap_if(c[2], c[4]);
    comp_swap_if(c[2], c[3]); comp_swap_if(c[0], c[3]); comp_swap_if(c[0], c[2]);
    comp_swap_if(c[1], c[4]); comp_swap_if(c[1], c[3]); comp_swap_if(c[1], c[2]);
}
template <> __device__ __forceinline__ void rank_sort<5, 3>(Comp<3> (&c)[5]) { net5(c); }
template <> __device__ __forceinline__ void rank_sort<5, 1>(Comp<1> (&c)[5]) { net5(c); }
template <> __device__ __forceinline__ void rank_sort<5, 4>(Comp<4> (&c)[5]) { net5(c); }

// Background test (§III.A) of the changed component at rank `rank` after
// the update: it is in B (the shortest rank prefix summing past T) unless the
// prefix before it already sums past T (prefix sums of non-negative weights
// do not decrease under rounding, so this equals rank >= B). A miss is
// foreground.
template <int M>
__device__ __forceinline__ int background_test(const float (&w)[M], int rank, bool matched,
                                               float T) {
    float acc = 0.f, before = 0.f;
#pragma unroll
    for (int r = 0; r < M - 1; ++r) {
        acc += w[r];
        if (r + 1 == rank)
            before = acc;
    }
    return (!matched || before > T) ? 1 : 0;
}
template <int M, int D>
__device__ __forceinline__ int background_test(const Comp<D> (&c)[M], int rank, bool matched,
                                               float T) {
    float w[M];
#pragma unroll
    for (int r = 0; r < M; ++r)
        w[r] = c[r].w;
    return background_test<M>(w, rank, matched, T);
}

// The update after the match (§III.A): weights, the changed component's mean
// and variance, re-ranking and the background test. hit: bit i set when
// component i lies within k standard deviations (the first set bit is the
// match); d2s: the squared distances. kJ >= 0: every lane of this call
// matched component kJ (the changed component is then known at compile time
// and needs no selects); kJ < 0: any outcome.
template <int M, int D, bool kOptions, int kJ>
__device__ __forceinline__ int mixture_update(Comp<D> (&c)[M], const float (&x)[D],
                                              const StreamPrm &p, uint32_t lanes, uint32_t hit,
                                              const float (&d2s)[M]) {
    const bool matched = kJ >= 0 || hit != 0u;
    const int jj = kJ >= 0 ? kJ : (matched ? __ffs(hit) - 1 : M - 1);
    float d2j = d2s[0];
    if (kOptions) {
#pragma unroll
        for (int i = 1; i < M; ++i)
            if (i == jj)
                d2j = d2s[i];
    }

    // The component that changes (matched, or the last-ranked on a miss),
    // gathered once.
    float muj[D], vj = c[0].v;
#pragma unroll
    for (int ch = 0; ch < D; ++ch)
        muj[ch] = c[0].mu[ch];
#pragma unroll
    for (int i = 1; i < M; ++i) {
        if (i == jj) {
            vj = c[i].v;
#pragma unroll
            for (int ch = 0; ch < D; ++ch)
                muj[ch] = c[i].mu[ch];
        }
    }

    // Weights decay; the matched one gains alpha, or the last-ranked one is
    // replaced on a miss; then renormalise. (Explicitly rounded operations:
    // no multiply-add contraction, so every path rounds alike.)
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        float w = __fmul_rn(c[i].w, p.oma);
        if (i == jj)
            w = matched ? __fadd_rn(w, p.alpha) : p.init_w;
        c[i].w = w;
        sum = __fadd_rn(sum, w);
    }
    const float inv = __fdividef(1.0f, sum); // within 2 ulp; the sum is near 1

    // Mean and variance of the changed component (the variance from the
    // squared distance to the new mean).
    if (matched) {
        float orho = p.oma, rho = p.alpha;
        if (kOptions)
            rho = match_rate<D>(p, d2j, vj, orho);
        float d2n = 0.f;
#pragma unroll
        for (int ch = 0; ch < D; ++ch) {
            muj[ch] = fmaf(orho, muj[ch], rho * x[ch]);
            const float df = x[ch] - muj[ch];
            d2n = fmaf(df, df, d2n);
        }
        vj = fmaxf(p.v_min, fmaf(orho, vj, rho * (kOptions ? var_sample<D>(p, d2n) : d2n)));
    } else {
#pragma unroll
        for (int ch = 0; ch < D; ++ch)
            muj[ch] = x[ch];
        vj = p.init_var;
    }
#pragma unroll
    for (int i = 0; i < M; ++i) {
        c[i].w *= inv;
        if (i == jj) {
#pragma unroll
            for (int ch = 0; ch < D; ++ch)
                c[i].mu[ch] = muj[ch];
            c[i].v = vj;
        }
        c[i].key = rank_key(c[i].w, c[i].v, i);
    }

    // Re-rank by w / sigma (stable), then the background test. When every
    // lane's components are already in non-increasing key order (the usual
    // case: a background pixel matches its best component and the others
    // decay by the same factor), the stable network would leave them as they
    // are, so the warp skips it and the changed component keeps its rank.
    bool sorted = true;
#pragma unroll
    for (int i = 1; i < M; ++i)
        sorted = sorted && !(c[i].key > c[i - 1].key);
    int rank = jj; // the changed component's rank after the update
    if (__any_sync(lanes, !sorted)) {
        rank_sort<M, D>(c);
#pragma unroll
        for (int r = 0; r < M; ++r)
            if ((c[r].key & 7u) == 7u - (uint32_t)jj) // its stored rank, from the key
                rank = r;
        if (kJ >= 0) // (the specialised path keeps its rank known where no sort ran)
            return background_test<M, D>(c, rank, matched, p.T);
    }
    return background_test<M, D>(c, rank, matched, p.T);
}

// One tick of one mixture at one pixel (§III.A). The components are in rank
// order on entry and on exit. Returns the stream's foreground bit. A warp
// skips the sorting network when it would change nothing; `lanes` is the set
// of lanes of the warp that make this same call, computed by the caller
// before the code diverged. Where every lane of the call matches its
// best-ranked component (the usual case for background pixels) a path
// specialised to that runs; it computes exactly what the general path does.
template <int M, int D, bool kOptions>
__device__ __forceinline__ int mixture_step(Comp<D> (&c)[M], const float (&x)[D],
                                            const StreamPrm &p, uint32_t lanes) {
    // Match: first component, in rank order, within k standard deviations
    // (bit i of hit: component i is within; the first set bit wins).
    uint32_t hit = 0u;
    float d2s[M];
#pragma unroll
    for (int i = 0; i < M; ++i) {
        float d2 = 0.f;
#pragma unroll
        for (int ch = 0; ch < D; ++ch) {
            const float df = x[ch] - c[i].mu[ch];
            d2 = fmaf(df, df, d2);
        }
        d2s[i] = d2;
        if (d2 < p.k2 * c[i].v)
            hit |= 1u << i;
    }
    if (__all_sync(lanes, hit & 1u))
        return mixture_update<M, D, kOptions, 0>(c, x, p, lanes, hit, d2s);
    return mixture_update<M, D, kOptions, -1>(c, x, p, lanes, hit, d2s);
}

// ------------------------------------- mixture step on what a pixel needs
// The same tick of one mixture without the whole state in hand. A tick
// changes every weight, and of the means and variances only those of the
// component that matched or was replaced, unless components change places.
// So it needs every weight and variance (the ranking) and the best-ranked
// component's mean, which the caller has loaded; the other means are loaded
// only in lanes that do not match the best-ranked component or whose
// components change places, and only what changed is stored: of 16 M values
// moved per pixel, 6 M + 10 remain for a background pixel. (Per-lane
// predicates: a warp moves the 32-byte sectors its lanes ask for. A lane that
// stores a mean or a variance has loaded that element, so a partly stored
// sector is one the L2 already holds.) Measured in FP32 against moving the
// whole state (HBM-bound at 100% of the copy bandwidth): one 1920x1080
// camera, M = 5, 101.1 -> 63.5 us per tick (DRAM reads 108 instead of 165
// bytes per pixel); 64 pooled cameras 2299 -> 1369 us. (Re-reading means
// where components change places, one plane at a time to save registers,
// measured 70.1 and 1390 us.)
//
// Io is where the state lives: load_means(m) fills the means m[1..] of this
// lane; put(r, mu, v) takes the new mean and variance at rank r
// (r known at compile time, only for ranks that changed). w, v: the weights
// (updated to the new ones, in rank order) and variances; mu: the best-ranked
// component's mean.
template <int M, int D, bool kOptions, int kJ, class Io>
__device__ __forceinline__ int ranked_update(Io &io, float (&w)[M], const float (&v)[M],
                                             float (&mu)[D], float (&m)[M][D],
                                             const float (&x)[D], const StreamPrm &p,
                                             uint32_t lanes, bool best, bool matched, int j,
                                             float d2j) {
    const int jj = kJ == 0 ? 0 : j; // the component that changes
    float vj = v[0];
    if (kJ != 0) {
#pragma unroll
        for (int i = 1; i < M; ++i)
            if (i == jj)
                vj = v[i];
    }
    // Weights decay; the matched one gains alpha, or the last-ranked one is
    // replaced on a miss; then renormalise. (Explicitly rounded operations:
    // no multiply-add contraction, so every path rounds alike.)
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        float wi = __fmul_rn(w[i], p.oma);
        if (i == jj)
            wi = matched ? __fadd_rn(wi, p.alpha) : p.init_w;
        w[i] = wi;
        sum = __fadd_rn(sum, wi);
    }
    const float inv = __fdividef(1.0f, sum); // within 2 ulp; the sum is near 1
    // Mean and variance of the changed component (the variance from the
    // squared distance to the new mean).
    if (matched) {
        float orho = p.oma, rho = p.alpha;
        if (kOptions)
            rho = match_rate<D>(p, d2j, vj, orho);
        float d2n = 0.f;
#pragma unroll
        for (int ch = 0; ch < D; ++ch) {
            mu[ch] = fmaf(orho, mu[ch], rho * x[ch]);
            const float df = x[ch] - mu[ch];
            d2n = fmaf(df, df, d2n);
        }
        vj = fmaxf(p.v_min, fmaf(orho, vj, rho * (kOptions ? var_sample<D>(p, d2n) : d2n)));
    } else {
#pragma unroll
        for (int ch = 0; ch < D; ++ch)
            mu[ch] = x[ch];
        vj = p.init_var;
    }
    // Re-rank by w / sigma (stable), then the background test. When every
    // lane's components are already in non-increasing key order (the usual
    // case), the stable network would leave them as they are, so the warp
    // skips it and the changed component keeps its rank.
    uint32_t key[M];
    bool sorted = true;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        w[i] *= inv;
        key[i] = rank_key(w[i], i == jj ? vj : v[i], i);
        if (i > 0)
            sorted = sorted && !(key[i] > key[i - 1]);
    }
    int rank = jj; // the changed component's rank after the update
    if (__any_sync(lanes, !sorted)) {
        if (!sorted && (kJ == 0 || best))
            io.load_means(m);
        Comp<D> c[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            c[i].key = key[i];
            c[i].w = w[i];
            c[i].v = i == jj ? vj : v[i];
#pragma unroll
            for (int ch = 0; ch < D; ++ch)
                c[i].mu[ch] = i == jj ? mu[ch] : m[i][ch];
        }
        rank_sort<M, D>(c);
#pragma unroll
        for (int r = 0; r < M; ++r) { // the stored rank is in the key
            const int id = 7 - (int)(c[r].key & 7u);
            if (id == jj)
                rank = r;
            w[r] = c[r].w;
            if (id == jj || id != r)
                io.put(r, c[r].mu, c[r].v);
        }
    } else {
#pragma unroll
        for (int r = 0; r < M; ++r)
            if (r == jj)
                io.put(r, mu, vj);
    }
    return background_test<M>(w, rank, matched, p.T);
}

// One tick of one mixture at one pixel (§III.A). The components are in rank
// order on entry and on exit. Returns the stream's foreground bit. lanes: the
// set of lanes of the warp that make this same call, computed by the caller
// before the code diverged. Two paths, which compute the same: one
// specialised to a match of the best-ranked component in every lane of the
// call (the usual case for background pixels), and the general one.
template <int M, int D, bool kOptions, class Io>
__device__ __forceinline__ int ranked_step(Io &io, float (&w)[M], const float (&v)[M],
                                           float (&mu)[D], const float (&x)[D],
                                           const StreamPrm &p, uint32_t lanes) {
    float d2 = 0.f;
#pragma unroll
    for (int ch = 0; ch < D; ++ch) {
        const float df = x[ch] - mu[ch];
        d2 = fmaf(df, df, d2);
    }
    const bool best = d2 < p.k2 * v[0];
    float m[M][D] = {};
    if (__all_sync(lanes, best))
        return ranked_update<M, D, kOptions, 0>(io, w, v, mu, m, x, p, lanes, true, true, 0, d2);
    bool matched = best;
    int jj = 0;
    if (!best) { // the first match, in rank order, within k standard deviations
        jj = M - 1; // replaced on a miss
        io.load_means(m);
#pragma unroll
        for (int ch = 0; ch < D; ++ch)
            m[0][ch] = mu[ch];
#pragma unroll
        for (int i = M - 1; i >= 1; --i) {
            float d2i = 0.f;
#pragma unroll
            for (int ch = 0; ch < D; ++ch) {
                const float df = x[ch] - m[i][ch];
                d2i = fmaf(df, df, d2i);
            }
            if (d2i < p.k2 * v[i]) {
                matched = true;
                jj = i;
                d2 = d2i;
#pragma unroll
                for (int ch = 0; ch < D; ++ch)
                    mu[ch] = m[i][ch];
            }
        }
    }
    return ranked_update<M, D, kOptions, -1>(io, w, v, mu, m, x, p, lanes, best, matched, jj, d2);
}

// List 1 (§III.C) on the low four bits of the per-pixel byte.
__device__ __forceinline__ uint32_t fuse_list1(int fgc, int fgd, uint32_t fb) {
    int F = (int)(fb & 1u);
    int cpt = (int)((fb >> 1) & 7u) - 3;
    if (fgc == fgd) {
        F = fgd;
        cpt = 0;
    } else if (cpt == 3) {
        F = fgc;
        cpt = 0;
    } else if (cpt == -3) {
        F = fgd;
        cpt = 0;
    } else if (F == fgc) {
        cpt += 1;
    } else {
        cpt -= 1;
    }
    return (fb & ~15u) | (uint32_t)F | ((uint32_t)(cpt + 3) << 1);
}

// Random bits for the weights of component i at padded pixel p when the
// view asks for stochastic rounding, else 0.
__device__ __forceinline__ uint32_t sr_weights(const CamView &cv, uint32_t p, int i) {
    if (!(cv.flags & kStochasticWeights))
        return 0u;
    const uint32_t r = sr_bits(cv.tick, p, (uint32_t)i);
    return r ? r : 1u;
}

// ------------------------------------------------------------ one pixel
// The first tick of a pixel in FP32 state: every component on the sample,
// w = 1/M; the depth model starts with the first reading (until then its
// planes are zero). The whole state is written; the foregrounds are 0.
template <int M, int kVariant>
__device__ __forceinline__ void first_pixel_f32(const CamView &cv, int64_t p, int64_t e0,
                                                const float (&xc)[3], uint32_t draw) {
    const float w0 = 1.0f / (float)M;
    const bool depth = kVariant != 2 && draw != 0u;
    float f[kFields];
    f[F_WC] = w0;
    f[F_MUR] = xc[0];
    f[F_MUG] = xc[1];
    f[F_MUB] = xc[2];
    f[F_VC] = cv.pc.init_var;
    f[F_WD] = depth ? w0 : 0.f;
    f[F_MUD] = kVariant == 2 ? (draw ? cv.depth_scale * (float)draw : 0.f) : (float)draw;
    f[F_VD] = depth ? cv.pd.init_var : 0.f;
    float *b = static_cast<float *>(cv.planes) + e0;
#pragma unroll
    for (int i = 0; i < M; ++i)
#pragma unroll
        for (int k = 0; k < kFields; ++k)
            b[(kFields * i + k) * kTile] = f[k];
    cv.fusion[p] = kVariant == 2 ? (uint8_t)0u
                                 : (uint8_t)fuse_list1(0, 0, depth ? kDepthStarted : 0u);
}

// Planes of one pixel's FP32 state as ranked_step's Io: D mean planes from
// field kMu, the variance plane kV. (D = 4: the fourth mean is the depth's.)
template <int M, int D, int kMu, int kV> struct PlanesF32 {
    float *b;
    static __device__ __forceinline__ constexpr int mean(int ch) {
        return ch < 3 ? kMu + ch : F_MUD;
    }
    __device__ __forceinline__ void load_means(float (&m)[M][D]) const {
#pragma unroll
        for (int i = 1; i < M; ++i)
#pragma unroll
            for (int ch = 0; ch < D; ++ch)
                m[i][ch] = b[(kFields * i + mean(ch)) * kTile];
    }
    __device__ __forceinline__ void put(int r, const float (&mu)[D], float v) const {
#pragma unroll
        for (int ch = 0; ch < D; ++ch)
            b[(kFields * r + mean(ch)) * kTile] = mu[ch];
        b[(kFields * r + kV) * kTile] = v;
    }
};

// FP32 state after the first tick. The loads that every lane needs come
// first, for both mixtures together.
template <int M, int kVariant>
__device__ __forceinline__ uint32_t tick_pixel_f32(const CamView &cv, int64_t p, int64_t e0,
                                                   const float (&xc)[3], uint32_t draw,
                                                   uint32_t lanes_c) {
    float *const b = static_cast<float *>(cv.planes) + e0;
    auto at = [b](int i, int f) -> float & { return b[(kFields * i + f) * kTile]; };
    float w[M], v[M];
#pragma unroll
    for (int i = 0; i < M; ++i) {
        w[i] = at(i, F_WC);
        v[i] = at(i, F_VC);
    }
    if constexpr (kVariant == 2) {
        // The augmentation alternative (§III.B): one mixture over R, G, B and
        // the scaled depth, stored in the colour planes plus the depth-mean
        // plane. A zero reading takes the best-ranked component's depth mean.
        float mu[4] = {at(0, F_MUR), at(0, F_MUG), at(0, F_MUB), at(0, F_MUD)};
        const float xa[4] = {xc[0], xc[1], xc[2], draw ? cv.depth_scale * (float)draw : mu[3]};
        PlanesF32<M, 4, F_MUR, F_VC> io = {b};
        const uint32_t f = (uint32_t)ranked_step<M, 4, true>(io, w, v, mu, xa, cv.pc, lanes_c);
#pragma unroll
        for (int r = 0; r < M; ++r)
            at(r, F_WC) = w[r];
        cv.fusion[p] = (uint8_t)f;
        return f | (f << 1) | (f << 2);
    } else {
        const uint32_t fb0 = cv.fusion[p];
        float mu[3] = {at(0, F_MUR), at(0, F_MUG), at(0, F_MUB)};
        float wd[M], vd[M], mud[1] = {at(0, F_MUD)};
#pragma unroll
        for (int i = 0; i < M; ++i) {
            wd[i] = at(i, F_WD);
            vd[i] = at(i, F_VD);
        }
        PlanesF32<M, 3, F_MUR, F_VC> colour = {b};
        const int fgc = ranked_step<M, 3, (kVariant != 0)>(colour, w, v, mu, xc, cv.pc, lanes_c);
#pragma unroll
        for (int r = 0; r < M; ++r)
            at(r, F_WC) = w[r];
        // The lanes that run the depth mixture: a reading, and a started model.
        uint32_t fb = fb0;
        const uint32_t lanes_d = __ballot_sync(lanes_c, draw != 0u && (fb & kDepthStarted));
        int fgd;
        if (draw == 0u) {
            fgd = fgc; // no reading: depth model untouched, depth answer = colour
        } else if (!(fb & kDepthStarted)) {
#pragma unroll
            for (int i = 0; i < M; ++i) {
                at(i, F_WD) = 1.0f / (float)M;
                at(i, F_MUD) = (float)draw;
                at(i, F_VD) = cv.pd.init_var;
            }
            fb |= kDepthStarted;
            fgd = 0;
        } else {
            const float xd[1] = {(float)draw};
            PlanesF32<M, 1, F_MUD, F_VD> depth = {b};
            fgd = ranked_step<M, 1, (kVariant != 0)>(depth, wd, vd, mud, xd, cv.pd, lanes_d);
#pragma unroll
            for (int r = 0; r < M; ++r)
                at(r, F_WD) = wd[r];
        }
        fb = fuse_list1(fgc, fgd, fb);
        if (fb != fb0)
            cv.fusion[p] = (uint8_t)fb;
        return (fb & 1u) | ((uint32_t)fgc << 1) | ((uint32_t)fgd << 2);
    }
}

// FP16/BF16 state: every group is loaded, and written back.
template <int M, int kVariant>
__device__ __forceinline__ uint32_t tick_pixel_f16(const CamView &cv, int64_t p, int64_t tb,
                                                   uint32_t t, const float (&xc)[3],
                                                   uint32_t draw, uint32_t lanes_c) {
    const float xd[1] = {(float)draw};
    const uint2 *const g = static_cast<const uint2 *>(cv.planes) + (tb >> 2) + t;
    auto store = [&](int i, const Fields &f) {
        const uint32_t sr = kVariant != 0 ? sr_weights(cv, (uint32_t)p, i) : 0u;
        store_fields_f16<kVariant != 0>(cv.planes, tb, t, i, f, sr);
    };
    if (kVariant == 2) {
        Comp<4> a[M];
        float xa[4] = {xc[0], xc[1], xc[2], cv.depth_scale * (float)draw};
        int fg;
        if (cv.first) {
            if (draw == 0u)
                xa[3] = 0.f;
#pragma unroll
            for (int i = 0; i < M; ++i) {
                a[i].w = 1.0f / (float)M;
                a[i].mu[0] = xa[0]; a[i].mu[1] = xa[1]; a[i].mu[2] = xa[2]; a[i].mu[3] = xa[3];
                a[i].v = cv.pc.init_var;
            }
            fg = 0;
        } else {
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const uint2 g0 = g[2 * i * kTile], g1 = g[(2 * i + 1) * kTile];
                a[i].w = bf16_lo(g0.x);
                const float2 rg = f16x2_unpack(g0.y), bv = f16x2_unpack(g1.x);
                a[i].mu[0] = rg.x; a[i].mu[1] = rg.y; a[i].mu[2] = bv.x;
                a[i].v = bv.y;
                a[i].mu[3] = f16x2_unpack(g1.y).x;
            }
            if (draw == 0u)
                xa[3] = a[0].mu[3];
            fg = mixture_step<M, 4, true>(a, xa, cv.pc, lanes_c);
        }
#pragma unroll
        for (int i = 0; i < M; ++i) // w_d and v_d are unused and read as zero
            store(i, {a[i].w, a[i].mu[0], a[i].mu[1], a[i].mu[2], a[i].v, 0.f, a[i].mu[3], 0.f});
        const uint32_t f = (uint32_t)fg;
        cv.fusion[p] = (uint8_t)f;
        return f | (f << 1) | (f << 2);
    }
    Comp<3> c[M];
    Comp<1> d[M];
    uint32_t fb;
    int fgc, fgd;
    if (cv.first) {
        fb = 0u;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            c[i].w = 1.0f / (float)M;
            c[i].mu[0] = xc[0]; c[i].mu[1] = xc[1]; c[i].mu[2] = xc[2];
            c[i].v = cv.pc.init_var;
            d[i].w = 0.f; d[i].mu[0] = 0.f; d[i].v = 0.f;
        }
        fgc = 0;
    } else {
        // The depth values stay packed (two registers per component instead
        // of three) while the colour mixture runs.
        fb = cv.fusion[p];
        uint32_t dw[M], dmv[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const uint2 g0 = g[2 * i * kTile], g1 = g[(2 * i + 1) * kTile];
            c[i].w = bf16_lo(g0.x);
            const float2 rg = f16x2_unpack(g0.y), bv = f16x2_unpack(g1.x);
            c[i].mu[0] = rg.x; c[i].mu[1] = rg.y; c[i].mu[2] = bv.x;
            c[i].v = bv.y;
            dw[i] = g0.x;
            dmv[i] = g1.y;
        }
        fgc = mixture_step<M, 3, (kVariant != 0)>(c, xc, cv.pc, lanes_c);
#pragma unroll
        for (int i = 0; i < M; ++i) {
            d[i].w = bf16_hi(dw[i]);
            const float2 mv = f16x2_unpack(dmv[i]);
            d[i].mu[0] = mv.x;
            d[i].v = mv.y;
        }
    }
    // The lanes that run the depth mixture: a reading, and a started model.
    const uint32_t lanes_d = __ballot_sync(lanes_c, draw != 0u && (fb & kDepthStarted));
    if (draw == 0u) {
        fgd = fgc; // no reading: depth model untouched, depth answer = colour
    } else if (!(fb & kDepthStarted)) {
#pragma unroll
        for (int i = 0; i < M; ++i) {
            d[i].w = 1.0f / (float)M;
            d[i].mu[0] = xd[0];
            d[i].v = cv.pd.init_var;
        }
        fb |= kDepthStarted;
        fgd = 0;
    } else {
        fgd = mixture_step<M, 1, (kVariant != 0)>(d, xd, cv.pd, lanes_d);
    }
    fb = fuse_list1(fgc, fgd, fb);
#pragma unroll
    for (int i = 0; i < M; ++i)
        store(i, {c[i].w, c[i].mu[0], c[i].mu[1], c[i].mu[2], c[i].v, d[i].w, d[i].mu[0], d[i].v});
    cv.fusion[p] = (uint8_t)fb;
    return (fb & 1u) | ((uint32_t)fgc << 1) | ((uint32_t)fgd << 2);
}

// p: padded linear pixel index (row * w_pad + x). Returns bit 0 fused label,
// bit 1 colour foreground, bit 2 depth foreground (all 0 for padding).
// kVariant: 0 the paper's method with the default readings; 1 the same with
// the learning-rate and variance options of StreamPrm.flags honoured; 2 the
// augmentation alternative (options honoured too).
template <int M, int PREC, int kVariant>
__device__ __forceinline__ uint32_t process_pixel(const CamView &cv, int64_t p) {
    const uint32_t p32 = (uint32_t)p;
    const uint32_t row = div_wpr(p32 >> 5, cv);
    const uint32_t x = p32 - row * (uint32_t)cv.w_pad;
    // Every caller enters with whole warps; the lanes on image pixels (not
    // row padding) are the ones that run the colour (or augmented) mixture.
    const uint32_t lanes_c = __ballot_sync(0xffffffffu, x < (uint32_t)cv.W);
    if (x >= (uint32_t)cv.W)
        return 0u;
    const int64_t q = (int64_t)row * cv.W + x;
    const float xc[3] = {(float)cv.rgb[3 * q], (float)cv.rgb[3 * q + 1],
                         (float)cv.rgb[3 * q + 2]};
    const uint32_t draw = cv.depth[q];
    // First element of the pixel's tile, and the pixel's column in it.
    const int64_t tb = (int64_t)(p32 / kTile) * (kFields * M * kTile);
    const uint32_t t = p32 % kTile;
    if constexpr (PREC == 0) {
        if (cv.first) {
            first_pixel_f32<M, kVariant>(cv, p, tb + t, xc, draw);
            return 0u;
        }
        return tick_pixel_f32<M, kVariant>(cv, p, tb + t, xc, draw, lanes_c);
    } else {
        return tick_pixel_f16<M, kVariant>(cv, p, tb, t, xc, draw, lanes_c);
    }
}

// All 32 lanes of the warp call this for 32 consecutive padded pixels
// starting at a multiple of 32 (word index wi).
__device__ __forceinline__ void write_mask_words(const CamView &cv, int64_t wi, uint32_t bits) {
    const uint32_t F = __ballot_sync(0xffffffffu, bits & 1u);
    const bool lane0 = (threadIdx.x & 31u) == 0u;
    if (lane0)
        cv.mask[wi] = F;
    if (cv.fg_rgb) { // uniform: the whole warp takes it or not
        const uint32_t fc = __ballot_sync(0xffffffffu, bits & 2u);
        if (lane0)
            cv.fg_rgb[wi] = fc;
    }
    if (cv.fg_d) {
        const uint32_t fd = __ballot_sync(0xffffffffu, bits & 4u);
        if (lane0)
            cv.fg_d[wi] = fd;
    }
}

} // namespace gmmdev
