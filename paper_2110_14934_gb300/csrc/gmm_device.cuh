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
//   FP16/BF16: planes of 4-byte pairs of one type, element (plane * kTile +
//         t) * 2 + slot: W_i = {w_c, w_d} at plane 2 i, V_i = {v_c, v_d} at
//         2 i + 1, RG_i = {mu_r, mu_g} at 2 M + 2 i, BD_i = {mu_b, mu_d} at
//         2 M + 2 i + 1: what every tick reads (all W and V, RG_0, BD_0) is
//         one contiguous block at the head of the tile, the other means
//         follow; a warp's access is one fully used 128-byte line, converted
//         by one packed instruction per pixel;
//   FP16/BF16 state that the caller owns (documented in gmm.h): two groups
//         of four 2-byte slots per component and pixel, group 0 = {w_c, w_d,
//         mu_r, mu_g}, group 1 = {mu_b, v_c, mu_d, v_d}, element ((2 i +
//         group) * kTile + t) * 4 + slot.
// The offsets of a pixel's values are compile-time constants from one base
// address, and a tile's whole state is one contiguous block that a single
// bulk copy moves. The List-1 byte of a pixel lives in a separate byte array
// indexed by p (n_tiles * kTile bytes).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

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
constexpr uint32_t kTinyVariance = 4u;  // StreamPrm.flags: a new variance may be denormal

// Storage of the state, as the kernels' PREC (CamView.prec).
enum { kF32 = 0, kF16 = 1, kF16Caller = 2 };

// Plane and slot of a field of component i in the FP16/BF16 pair layout.
__host__ __device__ constexpr int pair_plane(int M, int i, int f) {
    return f == F_WC || f == F_WD ? 2 * i
         : f == F_VC || f == F_VD ? 2 * i + 1
         : f == F_MUR || f == F_MUG ? 2 * M + 2 * i : 2 * M + 2 * i + 1;
}
__host__ __device__ constexpr int pair_slot(int f) {
    return f == F_WD || f == F_VD || f == F_MUG || f == F_MUD ? 1 : 0;
}

struct StreamPrm {
    float alpha, oma, k2, T, init_var, init_w, v_min;
    uint32_t flags; // kRhoEta | kVarPerChannel | kTinyVariance
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

// Everything one tick of one camera needs: a parameter of the single-camera
// kernel, one of up to 128 in those of the pooled kernels.
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
    int M, prec, first, flags; // prec: kF32..; flags: kStageInputs, kModeAugmented, kStochasticWeights
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

// Replace the low / high half of a pair, rounded like f16x2_pack_sat.
__device__ __forceinline__ uint32_t f16x2_set_lo(uint32_t pair, float lo) {
    return __byte_perm(f16x2_pack_sat(lo, lo), pair, 0x7610);
}
__device__ __forceinline__ uint32_t f16x2_set_hi(uint32_t pair, float hi) {
    return __byte_perm(f16x2_pack_sat(hi, hi), pair, 0x1054);
}

// ------------------------------------------------------------ mixture step
// Sort key of a component: the bits of w / sqrt(v) (a positive float, so its
// bits order like its value) with the low three bits replaced by 7 - the
// component's stored rank i. Comparing keys as unsigned integers orders by
// w / sigma and, between values that agree to 2^-20 relative (the same value
// included), puts the lower stored rank first: a total order, under which the
// network's result is the stable sort. (Two values that close lie well inside
// the 1e-5 margin at which a decision counts as near its threshold.)
// kNormalV: v is zero or a normal number, so the root needs no care for
// denormal ones (three instructions each; the result is the same).
template <bool kNormalV> __device__ __forceinline__ uint32_t rank_bits(float w, float v) {
    float r;
    if (kNormalV)
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    else
        r = rsqrtf(v);
    return __float_as_uint(w * r);
}
__device__ __forceinline__ uint32_t rank_key(uint32_t bits, int i) {
    return (bits & ~7u) | (7u - (uint32_t)i);
}
__device__ __forceinline__ uint32_t rank_key(float w, float v, int i) {
    return rank_key(rank_bits<false>(w, v), i);
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

// The matched component's new mean (in place) and variance (returned), from its
// variance v and the squared distance d2 to the old mean.
template <int D, bool kOptions>
__device__ __forceinline__ float moved_component(float (&mu)[D], float v, const float (&x)[D],
                                                 const StreamPrm &p, float d2) {
    float orho = p.oma, rho = p.alpha;
    if (kOptions)
        rho = match_rate<D>(p, d2, v, orho);
    float d2n = 0.f; // the variance follows the squared distance to the new mean
#pragma unroll
    for (int ch = 0; ch < D; ++ch) {
        mu[ch] = fmaf(orho, mu[ch], rho * x[ch]);
        const float df = x[ch] - mu[ch];
        d2n = fmaf(df, df, d2n);
    }
    return fmaxf(p.v_min, fmaf(orho, v, rho * (kOptions ? var_sample<D>(p, d2n) : d2n)));
}

// One tick of one mixture without the whole state in hand. A tick changes
// every weight, and of the means and variances only those of the component that
// matched or was replaced, unless components change places. So it needs every weight and variance (the ranking) and the best-ranked
// component's mean, which the caller has loaded; the other means are loaded
// only in lanes that do not match the best-ranked component or whose
// components change places, and only what changed is stored: of 16 M values
// moved per pixel, 6 M + 10 remain for a background pixel. (Per-lane
// predicates: a warp moves the 32-byte sectors its lanes ask for. A lane that
// stores a mean or a variance has loaded that element, so a partly stored
// sector is one the L2 already holds.) Measured in FP32 against moving the
// whole state (HBM-bound at 100% of the copy bandwidth), with the steps that
// followed: one 1920x1080 camera, M = 5, 101.1 -> 62.0 us per tick (DRAM reads
// 110 instead of 165 bytes per pixel); 64 pooled cameras 2294 -> 1266 us. In
// FP16/BF16: 54.7 -> 44.2 us, with the caller's layout (whose weights share a
// group with means) 1280x720, M = 4, with opening 25.5 -> 21.4 us. Frames in
// which every pixel misses cost a second trip: noise at 1920x1080, M = 5, FP32
// 101.5 -> 81.7 us, FP16/BF16 55.9 -> 58.0.
//
// Io is where the state lives: load_means(m, i0) fills this lane's stored
// means m[i0..]; put(r, mu, v) takes the new mean and variance at rank r
// (r known at compile time, only for ranks that changed). w, v: the weights
// (updated to the new ones, in rank order) and variances; mu: the best-ranked
// component's mean.
// Returns the stream's foreground bit. lanes: the set of lanes of the warp that
// make this same call, computed by the caller before the code diverged. Where
// every lane of the call matches its best-ranked component (the usual case
// for background pixels) the update is specialised to that; it computes
// exactly what the general one does. The ranking is one copy of code for both,
// and means are read again where components change places: with a ranking
// per path the pooled FP16/BF16 kernel, which holds a body per M, spent a
// third of its time on instruction fetch (24 cameras of odd sizes: 495 us
// against 404; FP32 1920x1080 63.5 against 64.7).
template <int M, int D, bool kOptions, bool kNormalV, class Io>
__device__ __forceinline__ int ranked_step(Io &io, float (&w)[M], float (&v)[M], float (&mu)[D],
                                           const float (&x)[D], const StreamPrm &p,
                                           uint32_t lanes) {
    float d2 = 0.f;
#pragma unroll
    for (int ch = 0; ch < D; ++ch) {
        const float df = x[ch] - mu[ch];
        d2 = fmaf(df, df, d2);
    }
    const bool best = d2 < p.k2 * v[0];
    const bool all_best = __all_sync(lanes, best);
    bool matched = best;
    int jj = 0; // the component that changes
    float sum;
    // Weights decay; the matched one gains alpha, or the last-ranked one is
    // replaced on a miss; then (below) renormalise. (Explicitly rounded
    // operations: no multiply-add contraction, so both paths round alike.)
    if (all_best) {
        w[0] = sum = __fadd_rn(__fmul_rn(w[0], p.oma), p.alpha);
#pragma unroll
        for (int i = 1; i < M; ++i) {
            w[i] = __fmul_rn(w[i], p.oma);
            sum = __fadd_rn(sum, w[i]);
        }
        v[0] = moved_component<D, kOptions>(mu, v[0], x, p, d2);
    } else {
        float vj = v[0];
        if (!best) { // the first match, in rank order, within k standard deviations
            jj = M - 1; // replaced on a miss
            float m[M][D];
            io.load_means(m, 1);
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
                    vj = v[i];
#pragma unroll
                    for (int ch = 0; ch < D; ++ch)
                        mu[ch] = m[i][ch];
                }
            }
        }
        if (matched) {
            vj = moved_component<D, kOptions>(mu, vj, x, p, d2);
        } else {
#pragma unroll
            for (int ch = 0; ch < D; ++ch)
                mu[ch] = x[ch];
            vj = p.init_var;
        }
        sum = 0.f;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            w[i] = __fmul_rn(w[i], p.oma);
            if (i == jj) {
                w[i] = matched ? __fadd_rn(w[i], p.alpha) : p.init_w;
                v[i] = vj;
            }
            sum = __fadd_rn(sum, w[i]);
        }
    }
    const float inv = __fdividef(1.0f, sum); // within 2 ulp; the sum is near 1
    // Re-rank by w / sigma (stable), then the background test. When every
    // lane's components are already in non-increasing key order (the usual
    // case), the stable network would leave them as they are, so the warp
    // skips it and the changed component keeps its rank.
    uint32_t bits[M];
    bool sorted = true;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        w[i] *= inv;
        bits[i] = rank_bits<kNormalV>(w[i], v[i]);
        if (i > 0) // rank_key(bits[i], i) > rank_key(bits[i - 1], i - 1)
            sorted = sorted && !(bits[i] > (bits[i - 1] | 7u));
    }
    int rank = jj; // the changed component's rank after the update
    if (__any_sync(lanes, !sorted)) {
        float m[M][D] = {};
        if (!sorted)
            io.load_means(m, 0);
        Comp<D> c[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            c[i].key = rank_key(bits[i], i);
            c[i].w = w[i];
            c[i].v = v[i];
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
    } else if (all_best) { // background: no weight comes before rank 0
        io.put(0, mu, v[0]);
        return 0;
    } else {
#pragma unroll
        for (int r = 0; r < M; ++r)
            if (r == jj)
                io.put(r, mu, v[r]);
    }
    return background_test<M>(w, rank, matched, p.T);
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
    __device__ __forceinline__ void load_means(float (&m)[M][D], int i0) const {
#pragma unroll
        for (int i = i0; i < M; ++i)
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
        const uint32_t f = (uint32_t)ranked_step<M, 4, true, false>(io, w, v, mu, xa, cv.pc, lanes_c);
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
        const int fgc = ranked_step<M, 3, (kVariant != 0), false>(colour, w, v, mu, xc, cv.pc, lanes_c);
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
            fgd = ranked_step<M, 1, (kVariant != 0), false>(depth, wd, vd, mud, xd, cv.pd, lanes_d);
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

// One pixel's FP16/BF16 state in the pair layout. Values stay packed until
// they are needed, and what did not change is never stored: the weights of
// every component always are, V and BD where either mixture changed them.
template <int M> struct PairsF16 {
    uint32_t *b; // the pixel's element of the tile's first plane
    uint32_t W[M], V[M], BD[M], RG0;
    bool loaded = false; // BD[1..] hold the stored values (or newer ones)
    uint32_t changed = 0u;

    __device__ __forceinline__ PairsF16(void *planes, int64_t tile, uint32_t t)
        : b(static_cast<uint32_t *>(planes) + tile * (4 * M * kTile) + t) {}
    __device__ __forceinline__ uint32_t &at(int plane) const { return b[plane * kTile]; }
    __device__ __forceinline__ void load() {
#pragma unroll
        for (int i = 0; i < M; ++i) {
            W[i] = at(2 * i);
            V[i] = at(2 * i + 1);
        }
        RG0 = at(2 * M);
        BD[0] = at(2 * M + 1);
    }
    __device__ __forceinline__ void load_bd() {
        if (loaded)
            return;
        loaded = true;
#pragma unroll
        for (int i = 1; i < M; ++i)
            BD[i] = at(2 * M + 2 * i + 1);
    }
    __device__ __forceinline__ float v_c(int i) const { return f16x2_unpack(V[i]).x; }
    __device__ __forceinline__ float v_d(int i) const { return f16x2_unpack(V[i]).y; }
    __device__ __forceinline__ float2 rg(int i) const {
        return f16x2_unpack(i == 0 ? RG0 : at(2 * M + 2 * i));
    }
    __device__ __forceinline__ float mu_b(int i) const { return f16x2_unpack(BD[i]).x; }
    __device__ __forceinline__ float mu_d(int i) const { return f16x2_unpack(BD[i]).y; }
    __device__ __forceinline__ void load_c() { load_bd(); }
    __device__ __forceinline__ void load_d() { load_bd(); }
    __device__ __forceinline__ void put_c(int r, const float *mu, float v) {
        at(2 * M + 2 * r) = f16x2_pack_sat(mu[0], mu[1]);
        BD[r] = f16x2_set_lo(BD[r], mu[2]);
        V[r] = f16x2_set_lo(V[r], v);
        changed |= 1u << r;
    }
    __device__ __forceinline__ void put_d(int r, float mu, float v) {
        BD[r] = f16x2_set_hi(BD[r], mu);
        V[r] = f16x2_set_hi(V[r], v);
        changed |= 1u << r;
    }
    __device__ __forceinline__ void clear_v_d() { // unused and read as zero (augmented mode)
#pragma unroll
        for (int i = 0; i < M; ++i) {
            if (V[i] >> 16) {
                V[i] &= 0xffffu;
                at(2 * i + 1) = V[i];
            }
        }
    }
    __device__ __forceinline__ void store(const uint32_t (&w)[M]) const {
#pragma unroll
        for (int i = 0; i < M; ++i)
            at(2 * i) = w[i];
        if (changed & 1u) {
            at(1) = V[0];
            at(2 * M + 1) = BD[0];
        }
        if (changed > 1u) {
#pragma unroll
            for (int i = 1; i < M; ++i) {
                if (changed >> i & 1u) {
                    at(2 * i + 1) = V[i];
                    at(2 * M + 2 * i + 1) = BD[i];
                }
            }
        }
    }
    // The first tick: component i whole.
    __device__ __forceinline__ void store_all(int i, uint32_t w, const float *mu, float v_c,
                                              float mu_d, float v_d) const {
        at(2 * i) = w;
        at(2 * i + 1) = f16x2_pack_sat(v_c, v_d);
        at(2 * M + 2 * i) = f16x2_pack_sat(mu[0], mu[1]);
        at(2 * M + 2 * i + 1) = f16x2_pack_sat(mu[2], mu_d);
    }
};

// The same in the caller-owned layout: the first group of a component (it
// holds the weights) is always stored, the second where it changed.
template <int M> struct GroupsF16 {
    uint2 *b;
    uint32_t W[M], RG[M], BV[M], DV[M]; // {w_c, w_d}, {mu_r, mu_g}, {mu_b, v_c}, {mu_d, v_d}
    uint32_t changed = 0u;

    __device__ __forceinline__ GroupsF16(void *planes, int64_t tile, uint32_t t)
        : b(static_cast<uint2 *>(planes) + tile * (2 * M * kTile) + t) {}
    __device__ __forceinline__ void load() {
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const uint2 g0 = b[2 * i * kTile], g1 = b[(2 * i + 1) * kTile];
            W[i] = g0.x;
            RG[i] = g0.y;
            BV[i] = g1.x;
            DV[i] = g1.y;
        }
    }
    __device__ __forceinline__ float v_c(int i) const { return f16x2_unpack(BV[i]).y; }
    __device__ __forceinline__ float v_d(int i) const { return f16x2_unpack(DV[i]).y; }
    __device__ __forceinline__ float2 rg(int i) const { return f16x2_unpack(RG[i]); }
    __device__ __forceinline__ float mu_b(int i) const { return f16x2_unpack(BV[i]).x; }
    __device__ __forceinline__ float mu_d(int i) const { return f16x2_unpack(DV[i]).x; }
    __device__ __forceinline__ void load_c() {}
    __device__ __forceinline__ void load_d() {}
    __device__ __forceinline__ void load_bd() {}
    __device__ __forceinline__ void put_c(int r, const float *mu, float v) {
        RG[r] = f16x2_pack_sat(mu[0], mu[1]);
        BV[r] = f16x2_pack_sat(mu[2], v);
        changed |= 1u << r;
    }
    __device__ __forceinline__ void put_d(int r, float mu, float v) {
        DV[r] = f16x2_pack_sat(mu, v);
        changed |= 1u << r;
    }
    __device__ __forceinline__ void clear_v_d() {
#pragma unroll
        for (int i = 0; i < M; ++i) {
            if (DV[i] >> 16) {
                DV[i] &= 0xffffu;
                changed |= 1u << i;
            }
        }
    }
    __device__ __forceinline__ void store(const uint32_t (&w)[M]) const {
#pragma unroll
        for (int i = 0; i < M; ++i)
            b[2 * i * kTile] = make_uint2(w[i], RG[i]);
        if (changed & 1u)
            b[kTile] = make_uint2(BV[0], DV[0]);
        if (changed > 1u) {
#pragma unroll
            for (int i = 1; i < M; ++i)
                if (changed >> i & 1u)
                    b[(2 * i + 1) * kTile] = make_uint2(BV[i], DV[i]);
        }
    }
    __device__ __forceinline__ void store_all(int i, uint32_t w, const float *mu, float v_c,
                                              float mu_d, float v_d) const {
        b[2 * i * kTile] = make_uint2(w, f16x2_pack_sat(mu[0], mu[1]));
        b[(2 * i + 1) * kTile] = make_uint2(f16x2_pack_sat(mu[2], v_c), f16x2_pack_sat(mu_d, v_d));
    }
};

// ranked_step's Io on either: the colour mixture, the depth mixture, the
// augmented one.
template <int M, class S> struct ColourF16 {
    S &s;
    __device__ __forceinline__ void load_means(float (&m)[M][3], int i0) {
        s.load_c();
#pragma unroll
        for (int i = i0; i < M; ++i) {
            const float2 rg = s.rg(i);
            m[i][0] = rg.x;
            m[i][1] = rg.y;
            m[i][2] = s.mu_b(i);
        }
    }
    __device__ __forceinline__ void put(int r, const float (&mu)[3], float v) { s.put_c(r, mu, v); }
};
template <int M, class S> struct DepthF16 {
    S &s;
    __device__ __forceinline__ void load_means(float (&m)[M][1], int i0) {
        s.load_d();
#pragma unroll
        for (int i = i0; i < M; ++i)
            m[i][0] = s.mu_d(i);
    }
    __device__ __forceinline__ void put(int r, const float (&mu)[1], float v) {
        s.put_d(r, mu[0], v);
    }
};
template <int M, class S> struct AugmentedF16 {
    S &s;
    __device__ __forceinline__ void load_means(float (&m)[M][4], int i0) {
        s.load_c();
#pragma unroll
        for (int i = i0; i < M; ++i) {
            const float2 rg = s.rg(i);
            m[i][0] = rg.x;
            m[i][1] = rg.y;
            m[i][2] = s.mu_b(i);
            m[i][3] = s.mu_d(i);
        }
    }
    __device__ __forceinline__ void put(int r, const float (&mu)[4], float v) {
        s.put_c(r, mu, v);
        s.put_d(r, mu[3], 0.f);
    }
};

// The two weights of component i as stored (stochastic rounding on request).
template <int kVariant>
__device__ __forceinline__ uint32_t pack_weights(const CamView &cv, uint32_t p, int i, float wc,
                                                 float wd) {
    const uint32_t sr = kVariant != 0 ? sr_weights(cv, p, i) : 0u;
    return (kVariant != 0 && sr) ? bf16x2_pack_sr(wc, wd, sr) : bf16x2_pack(wc, wd);
}

// FP16/BF16 state, the first tick (as first_pixel_f32).
template <int M, class S, int kVariant>
__device__ __forceinline__ void first_pixel_f16(const CamView &cv, int64_t p, S &s,
                                                const float (&xc)[3], uint32_t draw) {
    const float w0 = 1.0f / (float)M;
    const bool depth = kVariant != 2 && draw != 0u;
    const float z = kVariant == 2 ? (draw ? cv.depth_scale * (float)draw : 0.f) : (float)draw;
#pragma unroll
    for (int i = 0; i < M; ++i)
        s.store_all(i, pack_weights<kVariant>(cv, (uint32_t)p, i, w0, depth ? w0 : 0.f), xc,
                    cv.pc.init_var, z, depth ? cv.pd.init_var : 0.f);
    cv.fusion[p] = kVariant == 2 ? (uint8_t)0u
                                 : (uint8_t)fuse_list1(0, 0, depth ? kDepthStarted : 0u);
}

// FP16/BF16 state after the first tick. S: how the state is laid out.
template <int M, class S, int kVariant>
__device__ __forceinline__ uint32_t tick_pixel_f16(const CamView &cv, int64_t p, S &s,
                                                   const float (&xc)[3], uint32_t draw,
                                                   uint32_t lanes_c) {
    const uint32_t fb0 = kVariant == 2 ? 0u : cv.fusion[p];
    s.load();
    float w[M], v[M], wd[M];
    if constexpr (kVariant == 2) {
        s.clear_v_d();
#pragma unroll
        for (int i = 0; i < M; ++i) {
            w[i] = bf16_lo(s.W[i]);
            v[i] = s.v_c(i);
        }
        const float2 rg = s.rg(0);
        float mu[4] = {rg.x, rg.y, s.mu_b(0), s.mu_d(0)};
        const float xa[4] = {xc[0], xc[1], xc[2], draw ? cv.depth_scale * (float)draw : mu[3]};
        AugmentedF16<M, S> io = {s};
        const uint32_t f = (uint32_t)ranked_step<M, 4, true, false>(io, w, v, mu, xa, cv.pc, lanes_c);
        uint32_t packed[M]; // w_d is unused and reads as zero
#pragma unroll
        for (int i = 0; i < M; ++i)
            packed[i] = pack_weights<kVariant>(cv, (uint32_t)p, i, w[i], 0.f);
        s.store(packed);
        cv.fusion[p] = (uint8_t)f;
        return f | (f << 1) | (f << 2);
    } else {
        int fgc, fgd;
        {
#pragma unroll
            for (int i = 0; i < M; ++i) {
                w[i] = bf16_lo(s.W[i]);
                v[i] = s.v_c(i);
            }
            const float2 rg = s.rg(0);
            float mu[3] = {rg.x, rg.y, s.mu_b(0)};
            ColourF16<M, S> io = {s};
            fgc = ranked_step<M, 3, (kVariant != 0), (kVariant == 0)>(io, w, v, mu, xc, cv.pc, lanes_c);
        }
        // The lanes that run the depth mixture: a reading, and a started model.
        uint32_t fb = fb0;
        const uint32_t lanes_d = __ballot_sync(lanes_c, draw != 0u && (fb & kDepthStarted));
#pragma unroll
        for (int i = 0; i < M; ++i)
            wd[i] = bf16_hi(s.W[i]);
        if (draw == 0u) {
            fgd = fgc; // no reading: depth model untouched, depth answer = colour
        } else if (!(fb & kDepthStarted)) {
            s.load_bd();
#pragma unroll
            for (int i = 0; i < M; ++i) {
                wd[i] = 1.0f / (float)M;
                s.put_d(i, (float)draw, cv.pd.init_var);
            }
            fb |= kDepthStarted;
            fgd = 0;
        } else {
#pragma unroll
            for (int i = 0; i < M; ++i)
                v[i] = s.v_d(i);
            const float xd[1] = {(float)draw};
            float mu[1] = {s.mu_d(0)};
            DepthF16<M, S> io = {s};
            fgd = ranked_step<M, 1, (kVariant != 0), (kVariant == 0)>(io, wd, v, mu, xd, cv.pd, lanes_d);
        }
        fb = fuse_list1(fgc, fgd, fb);
        uint32_t packed[M];
#pragma unroll
        for (int i = 0; i < M; ++i)
            packed[i] = pack_weights<kVariant>(cv, (uint32_t)p, i, w[i], wd[i]);
        s.store(packed);
        if (fb != fb0)
            cv.fusion[p] = (uint8_t)fb;
        return (fb & 1u) | ((uint32_t)fgc << 1) | ((uint32_t)fgd << 2);
    }
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
    // The pixel's state tile, and its column in it.
    const int64_t tile = p32 / kTile;
    const uint32_t t = p32 % kTile;
    if constexpr (PREC == kF32) {
        const int64_t e0 = tile * (kFields * M * kTile) + t;
        if (cv.first) {
            first_pixel_f32<M, kVariant>(cv, p, e0, xc, draw);
            return 0u;
        }
        return tick_pixel_f32<M, kVariant>(cv, p, e0, xc, draw, lanes_c);
    } else {
        using S = std::conditional_t<PREC == kF16, PairsF16<M>, GroupsF16<M>>;
        S s(cv.planes, tile, t);
        if (cv.first) {
            first_pixel_f16<M, S, kVariant>(cv, p, s, xc, draw);
            return 0u;
        }
        return tick_pixel_f16<M, S, kVariant>(cv, p, s, xc, draw, lanes_c);
    }
}

// Move what a tick always reads of a warp's 32 pixels (p: this lane's padded
// pixel, consecutive from a multiple of 32) closer, one 128-byte line per
// lane: a hint, which reads nothing itself.
template <int M, int PREC, int V>
__device__ __forceinline__ void prefetch_pixels(const CamView &cv, int64_t p) {
    const uint32_t p32 = (uint32_t)p, lane = p32 & 31u, t = p32 % kTile - lane;
    const char *tile = static_cast<const char *>(cv.planes) +
                       (int64_t)(p32 / kTile) * (kFields * M * kTile * (PREC == kF32 ? 4 : 2));
    uint32_t off;
    constexpr uint32_t kLines = PREC == kF32 ? 4 * M + 4 : PREC == kF16 ? 2 * M + 2 : 4 * M;
    if (PREC == kF32) { // w_c, v_c, w_d, v_d of every component, the means of component 0
        const uint32_t i = lane < 4 * M ? lane >> 2 : 0u;
        const uint32_t f = (lane < 4 * M ? 0x7540u : 0x6321u) >> (4 * (lane & 3u)) & 15u;
        off = ((kFields * i + f) * kTile + t) * 4;
    } else if (PREC == kF16) { // the planes at the head of the tile
        off = (lane * kTile + t) * 4;
    } else { // every group, two lines each
        off = ((lane >> 1) * kTile + t) * 8 + (lane & 1u) * 128;
    }
    const bool unused = PREC == kF32 && V == 2 && lane < 4 * M && (lane & 2u); // w_d, v_d
    if (lane < kLines && !unused)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(tile + off));
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
