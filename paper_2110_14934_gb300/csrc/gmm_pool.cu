// Multi-camera pool: resident per-camera models, one persistent launch per
// tick over every camera with a submitted frame, and an autotuner for the
// launch shape.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <new>
#include <string>
#include <utility>
#include <vector>

#include "gmm.h"
#include "gmm_common.h"
#include "gmm_internal.h"
#include "gmm_pool_plan.h"

using gmmdev::CamView;
using namespace gmmlib;

namespace {

struct PoolCam {
    bool used = false;
    gmm_config cfg{};
    Layout L{};
    void *arena = nullptr;
    int initialized = 0;
    uint32_t ticks = 0; // ticks taken (seeds stochastic rounding)
    bool submitted = false;
    const uint8_t *rgb = nullptr;
    const uint16_t *depth = nullptr;
    uint32_t *mask = nullptr, *fgr = nullptr, *fgd = nullptr;
};

static_assert(kLaunchCams == gmmhost::kPoolViews, "a launch's cameras fit its parameters");

int chunk_pixels(int prec) { return prec == 0 ? 32 : 64; }

// Online tuning: real ticks cycle through candidate launch shapes; a trial
// tick is timed on the pool's stream from its start to the start of the
// next tick (the tick period), so a shape is also charged for what its
// kernel delays in the work queued before the next tick (uploads of the next
// frames sharing HBM with it, in a pipeline). Two rounds: when every
// candidate has run its ticks, the kFinalists shapes with the lowest median
// periods run again with twice the ticks each, and the lowest median of
// that second round is kept (shapes a few percent apart are told apart
// without giving every candidate the longer run).
struct Trial {
    int cand = -1;
    cudaEvent_t a = nullptr, b = nullptr;
};
constexpr int kFinalists = 4;
struct Tuning {
    bool active = false;
    bool final_round = false;
    bool named = false; // cands are the shapes that run (set by the first trial tick)
    int per_shape = 0, issued = 0;
    std::vector<Shape> cands;
    Trial open;                 // the last trial tick, until the next tick starts
    std::vector<Trial> pending; // closed trials not yet read
    std::vector<std::vector<float>> ms;
};

} // namespace

namespace gmmhost {
int pool_max_ctas_per_sm(int prec, int threads);
}

struct gmm_pool {
    size_t budget = 0, used_bytes = 0;
    int prec = 0, max_cams = 0, device = 0;
    std::vector<PoolCam> cams;
    cudaStream_t stream = nullptr;
    // The last work on the pool's state: whether there is any, whether it went
    // to the legacy stream, and else an event behind it (order_before).
    bool worked = false, worked_on_legacy = false;
    cudaEvent_t ev_work = nullptr;
    cudaMemPool_t mempool = nullptr;   // cameras' state; keeps freed memory mapped
    cudaError_t sticky = cudaSuccess;
    int threads = 128, ctas_per_sm = 0, tile_pixels = 2048; // ctas_per_sm < 0: flat form
    // Tile counters, two sets of kmax (one per launch of a tick): a tick
    // uses set `parity` and its launches zero the other set for the next.
    int *d_counters = nullptr;
    int kmax = 1, parity = 0; // kmax: launches a tick may take
    std::vector<TickCam> tick_cams;      // the tick's cameras, in order of M
    std::vector<LaunchPlan> plan;        // its launches (at most kmax)
    std::vector<gmmhost::PoolArgs> args; // and their arguments
    bool prefetch = true; // FP16/BF16: L2 prefetch in the persistent form
    Tuning tune;
    int occupancy[9] = {};  // resident pool CTAs per SM, by block size / 32
    int sms = 0;
};

// CTAs of the persistent form: resident CTAs per SM of the pool kernel for a
// block size (queried once per block size) times the SM count (queried once).
static int blocks_for(gmm_pool *p, int threads, int ctas_per_sm) {
    int &max_per_sm = p->occupancy[threads / 32];
    if (max_per_sm == 0)
        max_per_sm = gmmhost::pool_max_ctas_per_sm(p->prec, threads);
    if (p->sms == 0)
        p->sms = gmmhost::num_sms();
    int per_sm = ctas_per_sm;
    if (per_sm <= 0 || per_sm > max_per_sm)
        per_sm = max_per_sm;
    if (per_sm < 1)
        per_sm = 1;
    return p->sms * per_sm;
}

// The cameras with a submitted frame, in order of M: the flat form launches per
// M; in the persistent form the CTAs that run together then run one M's body of
// code (with the cameras mixed, the bodies of all three evict each other from
// the instruction caches), and the longest tiles come first.
static const std::vector<TickCam> &submitted_cams(gmm_pool *p) {
    p->tick_cams.clear();
    for (int m : {5, 4, 3})
        for (size_t i = 0; i < p->cams.size(); ++i) {
            const PoolCam &c = p->cams[i];
            if (c.used && c.submitted && c.cfg.M == m)
                p->tick_cams.push_back({(int)i, m, c.L.n_pad});
        }
    return p->tick_cams;
}

// Candidate launch shapes: block sizes, full or half residency, tile sizes
// of the persistent form. (The flat form is left to an explicit choice: it
// is the faster one for FP32 state with every input already in device
// memory, but host uploads that run beside it slow it far more than they
// slow the persistent form, and ticks timed without such uploads cannot
// tell.) A small tick runs smaller tiles than the larger of these
// (launch_tile): distinct_shapes leaves those that differ on the tick at hand.
static std::vector<Shape> tuning_candidates(const gmm_pool *p) {
    std::vector<Shape> out;
    const int cand_threads[] = {64, 128, 256};
    const int cand_tiles[] = {256, 512, 1024, 2048, 8192};
    for (int t : cand_threads) {
        const int max_c = gmmhost::pool_max_ctas_per_sm(p->prec, t);
        const int cand_c[2] = {max_c, max_c > 1 ? max_c / 2 : 0};
        for (int c : cand_c)
            if (c >= 1)
                for (int tp : cand_tiles)
                    out.push_back({t, c, tp});
    }
    return out;
}

static float median(std::vector<float> v) {
    if (v.empty())
        return -1.f;
    std::sort(v.begin(), v.end());
    return v[v.size() / 2];
}

// Read the finished trials; when all are in, keep the best shape.
static int tuning_poll(gmm_pool *p, bool block) {
    Tuning &tu = p->tune;
    if (!tu.active)
        return GMM_OK;
    size_t k = 0;
    for (; k < tu.pending.size(); ++k) {
        Trial &tr = tu.pending[k];
        cudaError_t e = block ? cudaEventSynchronize(tr.b) : cudaEventQuery(tr.b);
        if (e == cudaErrorNotReady)
            break;
        float ms = 0.f;
        if (e == cudaSuccess)
            e = cudaEventElapsedTime(&ms, tr.a, tr.b);
        cudaEventDestroy(tr.a);
        cudaEventDestroy(tr.b);
        if (e != cudaSuccess) {
            tu.pending.erase(tu.pending.begin(), tu.pending.begin() + (long)k + 1);
            return cuda_fail(&p->sticky, e, "gmm_pool tuning");
        }
        tu.ms[tr.cand].push_back(ms);
    }
    tu.pending.erase(tu.pending.begin(), tu.pending.begin() + (long)k);
    const int total = (int)tu.cands.size() * tu.per_shape;
    if (tu.issued < total || tu.open.a || !tu.pending.empty())
        return GMM_OK;
    std::vector<std::pair<float, int>> order; // (median period, candidate); untimed last
    for (size_t c = 0; c < tu.cands.size(); ++c) {
        const float m = median(tu.ms[c]);
        order.push_back({m >= 0.f ? m : 3.4e38f, (int)c});
    }
    std::stable_sort(order.begin(), order.end(),
                     [](const std::pair<float, int> &x, const std::pair<float, int> &y) {
                         return x.first < y.first;
                     });
    if (!tu.final_round && (int)tu.cands.size() > kFinalists) {
        std::vector<Shape> fin;
        for (int i = 0; i < kFinalists; ++i)
            fin.push_back(tu.cands[order[i].second]);
        tu.cands = fin;
        tu.ms.assign(fin.size(), {});
        tu.per_shape *= 2;
        tu.issued = 0;
        tu.final_round = true;
        return GMM_OK; // the next ticks run the finalists
    }
    const int best = order[0].second;
    p->threads = tu.cands[best].threads;
    p->ctas_per_sm = tu.cands[best].ctas;
    p->tile_pixels = tu.cands[best].tile;
    tu.active = false;
    return GMM_OK;
}

// Work on a pool's state and tile counters (ticks, admissions, releases, state
// reads) follows the pool's work before it, on whatever stream that was. The
// handles do not say whether it was the same one: cudaStreamPerThread is
// another stream in every thread, and a destroyed stream's handle may come back
// for a new one while the old one's work is still queued. So work on any stream
// but the legacy one leaves an event behind it, and the next work waits for it
// (ticks on one created stream, with and without that wait: 12 cameras of
// 320x240 20.2-20.4 and 20.4-20.6 us, 24 FP16/BF16 cameras of odd sizes 275 and
// 275; the event alone parts them). The legacy stream is one per device and always
// exists: work that stays on it needs no event, which would cost consecutive
// ticks their programmatic overlap, and it can be recorded later.
static cudaError_t order_before(gmm_pool *p) {
    if (!p->worked || (p->worked_on_legacy && !p->stream))
        return cudaSuccess;
    cudaError_t e = p->worked_on_legacy ? cudaEventRecord(p->ev_work, nullptr) : cudaSuccess;
    return e == cudaSuccess ? cudaStreamWaitEvent(p->stream, p->ev_work, 0) : e;
}

static cudaError_t order_after(gmm_pool *p) {
    p->worked = true;
    p->worked_on_legacy = !p->stream;
    return p->stream ? cudaEventRecord(p->ev_work, p->stream) : cudaSuccess;
}

// The host waits for the pool's last work, without using its stream.
static cudaError_t wait_for_work(const gmm_pool *p) {
    if (!p->worked)
        return cudaSuccess;
    return p->worked_on_legacy ? cudaStreamSynchronize(nullptr) : cudaEventSynchronize(p->ev_work);
}

// Launch the planned launches.
static cudaError_t launch_tick(gmm_pool *p, bool all_variants) {
    const bool flat = p->ctas_per_sm < 0;
    const int warps = p->threads / 32;
    cudaError_t e = order_before(p);
    for (size_t li = 0; li < p->plan.size() && e == cudaSuccess; ++li) {
        const gmmhost::PoolArgs &a = p->args[li];
        const int blocks = flat ? (int)((a.n_tiles + warps - 1) / warps)
                                : blocks_for(p, p->threads, p->ctas_per_sm);
        e = gmmhost::launch_pool_tick_impl(a, p->threads, blocks, p->prec, all_variants, flat,
                                           p->plan[li].m, p->prefetch, p->stream);
    }
    if (e == cudaSuccess)
        e = order_after(p);
    return e;
}

// One tick over the submitted cameras. clear: drop the submissions and mark
// the cameras initialised afterwards (false while autotuning).
static int pool_tick_impl(gmm_pool *p, bool clear) {
    const std::vector<TickCam> &cams = submitted_cams(p);
    // An online-tuning trial sets its launch shape first: the launches and
    // their tiles depend on it.
    Tuning &tu = p->tune;
    if (clear && tu.active && !tu.named) {
        tu.cands = distinct_shapes(tu.cands, cams, [&](const Shape &s) {
            return blocks_for(p, s.threads, s.ctas);
        });
        tu.ms.assign(tu.cands.size(), {});
        tu.named = true;
    }
    const bool trial = clear && tu.active && tu.issued < (int)tu.cands.size() * tu.per_shape;
    Trial tr{};
    if (trial) {
        // round-robin over the candidates, so drift in the frames spreads evenly
        tr.cand = tu.issued % (int)tu.cands.size();
        p->threads = tu.cands[tr.cand].threads;
        p->ctas_per_sm = tu.cands[tr.cand].ctas;
        p->tile_pixels = tu.cands[tr.cand].tile;
    }
    // The launches' arguments; tiles, or in the flat form one chunk per warp.
    const bool flat = p->ctas_per_sm < 0;
    const Shape shape = {p->threads, p->ctas_per_sm,
                         flat ? chunk_pixels(p->prec) : p->tile_pixels};
    plan_launches(cams, shape, flat ? 0 : blocks_for(p, p->threads, p->ctas_per_sm), p->plan);
    int *cur = p->d_counters + p->parity * p->kmax;
    int *next = p->d_counters + (1 - p->parity) * p->kmax;
    bool all_variants = false; // some camera needs the options or the augmented mixture
    for (size_t li = 0; li < p->plan.size(); ++li) {
        const LaunchPlan &l = p->plan[li];
        gmmhost::PoolArgs &a = p->args[li];
        int64_t tiles = 0;
        for (int j = 0; j < l.count; ++j) {
            const PoolCam &c = p->cams[cams[l.first + j].slot];
            a.views[j] = make_view(c.cfg, c.L, c.arena, c.rgb, c.depth, c.mask, c.fgr, c.fgd,
                                   c.initialized ? 0 : 1, c.ticks);
            all_variants = all_variants || gmmhost::view_variant(a.views[j]) != 0;
            a.tile_begin[j] = tiles;
            tiles += (c.L.n_pad + l.unit - 1) / l.unit;
        }
        a.tile_begin[l.count] = tiles;
        a.n_jobs = l.count;
        a.n_tiles = tiles;
        a.tile_pixels = l.unit;
        a.counter = cur + li;
        a.reset = next;
        a.n_reset = p->kmax;
    }
    cudaError_t e = cudaSuccess;
    if (clear && tu.active && tu.open.a) { // this tick's start ends the last trial's period
        e = cudaEventCreate(&tu.open.b);
        if (e == cudaSuccess)
            e = cudaEventRecord(tu.open.b, p->stream);
        if (e != cudaSuccess)
            return cuda_fail(&p->sticky, e, "gmm_pool_tick tuning");
        tu.pending.push_back(tu.open);
        tu.open = Trial();
    }
    if (trial) {
        e = cudaEventCreate(&tr.a);
        if (e == cudaSuccess)
            e = cudaEventRecord(tr.a, p->stream);
        if (e != cudaSuccess) {
            if (tr.a)
                cudaEventDestroy(tr.a);
            return cuda_fail(&p->sticky, e, "gmm_pool_tick tuning");
        }
        tu.open = tr;
        ++tu.issued;
    }
    e = launch_tick(p, all_variants);
    if (e != cudaSuccess)
        return cuda_fail(&p->sticky, e, "gmm_pool_tick");
    p->parity ^= 1;
    if (clear) {
        for (PoolCam &c : p->cams) {
            if (c.used && c.submitted) {
                c.initialized = 1;
                c.ticks += 1;
                c.submitted = false;
            }
        }
    }
    return tuning_poll(p, false);
}

static bool valid_cam(const gmm_pool *p, int cam) {
    return p && cam >= 0 && cam < (int)p->cams.size() && p->cams[cam].used;
}

extern "C" {

gmm_pool_t *gmm_pool_create(size_t budget_bytes, int precision, int max_cams) {
    if (precision != GMM_PREC_F32 && precision != GMM_PREC_F16) {
        fail(GMM_EINVAL, "gmm_pool_create: bad precision");
        return nullptr;
    }
    if (max_cams < 1 || max_cams > 65536) {
        fail(GMM_EINVAL, "gmm_pool_create: max_cams must be in [1, 65536]");
        return nullptr;
    }
    gmm_pool *p = new (std::nothrow) gmm_pool();
    if (!p) {
        fail(GMM_ENOMEM, "gmm_pool_create: host allocation failed");
        return nullptr;
    }
    p->budget = budget_bytes;
    p->prec = precision;
    p->max_cams = max_cams;
    // one launch per kLaunchCams cameras, plus one per M group in the flat form
    p->kmax = (max_cams + kLaunchCams - 1) / kLaunchCams + 2;
    try {
        p->cams.resize((size_t)max_cams);
        p->tick_cams.reserve((size_t)max_cams);
        p->plan.reserve((size_t)p->kmax);
        p->args.resize((size_t)p->kmax);
    } catch (const std::bad_alloc &) {
        fail(GMM_ENOMEM, "gmm_pool_create: host allocation failed");
        delete p;
        return nullptr;
    }
    cudaError_t e = cudaGetDevice(&p->device);
    if (e == cudaSuccess)
        e = cudaEventCreateWithFlags(&p->ev_work, cudaEventDisableTiming);
    if (e == cudaSuccess)
        e = cudaMalloc(&p->d_counters, sizeof(int) * 2 * (size_t)p->kmax);
    if (e == cudaSuccess)
        e = cudaMemset(p->d_counters, 0, sizeof(int) * 2 * (size_t)p->kmax);
    if (e == cudaSuccess)
        e = make_retaining_pool(p->device, budget_bytes ? (uint64_t)budget_bytes : UINT64_MAX,
                                &p->mempool);
    if (e != cudaSuccess) {
        fail(e == cudaErrorMemoryAllocation ? GMM_ENOMEM : GMM_ECUDA,
             std::string("gmm_pool_create: ") + cudaGetErrorString(e));
        cudaGetLastError();
        gmm_pool_destroy(p);
        return nullptr;
    }
    return p;
}

int gmm_pool_admit(gmm_pool_t *p, const gmm_config *cfg) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_admit: null pool");
    const std::string msg = check_config(cfg);
    if (!msg.empty())
        return fail(GMM_EINVAL, "gmm_pool_admit: " + msg);
    if (cfg->precision != p->prec)
        return fail(GMM_EINVAL, "gmm_pool_admit: precision differs from the pool's");
    if (cfg->morph_open)
        return fail(GMM_EINVAL, "gmm_pool_admit: morph_open is not supported in a pool");
    const Layout L = make_layout(cfg->H, cfg->W, cfg->M, cfg->precision);
    if (p->budget && p->used_bytes + L.total > p->budget)
        return fail(GMM_EBUDGET, "gmm_pool_admit: state budget exhausted");
    int slot = -1;
    for (int i = 0; i < (int)p->cams.size(); ++i)
        if (!p->cams[i].used) {
            slot = i;
            break;
        }
    if (slot < 0)
        return fail(GMM_ENOMEM, "gmm_pool_admit: every slot is taken");
    DeviceGuard g(p->device);
    void *arena = nullptr;
    cudaError_t e = order_before(p);
    if (e == cudaSuccess)
        e = cudaMallocFromPoolAsync(&arena, L.total, p->mempool, p->stream);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(arena, 0, L.total, p->stream);
    if (e == cudaSuccess)
        e = order_after(p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        if (arena)
            cudaFreeAsync(arena, p->stream);
        return fail(e == cudaErrorMemoryAllocation ? GMM_ENOMEM : GMM_ECUDA,
                    std::string("gmm_pool_admit: ") + cudaGetErrorString(e));
    }
    PoolCam &c = p->cams[slot];
    c = PoolCam();
    c.used = true;
    c.cfg = *cfg;
    c.L = L;
    c.arena = arena;
    p->used_bytes += L.total;
    return slot;
}

int gmm_pool_reserve(gmm_pool_t *p, size_t bytes) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_reserve: null pool");
    if (p->budget && bytes > p->budget)
        bytes = p->budget;
    DeviceGuard g(p->device);
    const cudaError_t e = reserve_in_pool(p->mempool, bytes, p->stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(e == cudaErrorMemoryAllocation ? GMM_ENOMEM : GMM_ECUDA,
                    std::string("gmm_pool_reserve: ") + cudaGetErrorString(e));
    }
    return GMM_OK;
}

int gmm_pool_release(gmm_pool_t *p, int cam) {
    if (!valid_cam(p, cam))
        return fail(GMM_EINVAL, "gmm_pool_release: unknown camera");
    DeviceGuard g(p->device);
    PoolCam &c = p->cams[cam];
    // Stream-ordered free: queued ticks that use the state run first.
    cudaError_t e = order_before(p);
    if (e == cudaSuccess)
        e = cudaFreeAsync(c.arena, p->stream);
    if (e == cudaSuccess)
        e = order_after(p);
    p->used_bytes -= c.L.total;
    c = PoolCam();
    if (e != cudaSuccess)
        return cuda_fail(&p->sticky, e, "gmm_pool_release");
    return GMM_OK;
}

int gmm_pool_submit(gmm_pool_t *p, int cam, const uint8_t *rgb8, const uint16_t *depth16,
                    uint32_t *mask_out, uint32_t *fg_rgb_out, uint32_t *fg_d_out) {
    if (!valid_cam(p, cam))
        return fail(GMM_EINVAL, "gmm_pool_submit: unknown camera");
    const std::string msg = check_frame_ptrs(rgb8, depth16, mask_out, fg_rgb_out, fg_d_out);
    if (!msg.empty())
        return fail(GMM_EINVAL, "gmm_pool_submit: " + msg);
    PoolCam &c = p->cams[cam];
    c.submitted = true;
    c.rgb = rgb8;
    c.depth = depth16;
    c.mask = mask_out;
    c.fgr = fg_rgb_out;
    c.fgd = fg_d_out;
    return GMM_OK;
}

int gmm_pool_submit_many(gmm_pool_t *p, int n, const int *cams, const uint8_t *const *rgb8,
                         const uint16_t *const *depth16, uint32_t *const *mask_out) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_submit_many: null pool");
    if (n < 0 || (n > 0 && (!cams || !rgb8 || !depth16 || !mask_out)))
        return fail(GMM_EINVAL, "gmm_pool_submit_many: bad arrays");
    for (int i = 0; i < n; ++i) {
        const int rc = gmm_pool_submit(p, cams[i], rgb8[i], depth16[i], mask_out[i], nullptr,
                                       nullptr);
        if (rc != GMM_OK)
            return rc;
    }
    return GMM_OK;
}

int gmm_pool_inject_cuda_error(gmm_pool_t *p, int cuda_error) {
    if (!p || cuda_error == 0)
        return fail(GMM_EINVAL, "gmm_pool_inject_cuda_error: null pool or zero error code");
    if (p->sticky == cudaSuccess)
        p->sticky = static_cast<cudaError_t>(cuda_error);
    return GMM_OK;
}

int gmm_pool_tick(gmm_pool_t *p) {
    TraceRange tr("gmm_pool_tick");
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_tick: null pool");
    if (p->sticky != cudaSuccess)
        return fail(GMM_ECUDA, std::string("gmm_pool_tick: earlier CUDA failure: ") +
                                   cudaGetErrorString(p->sticky));
    DeviceGuard g(p->device);
    if (submitted_cams(p).empty())
        return GMM_OK; // nothing to launch, on a capturing stream too
    // A captured tick would replay with this tick's tile counters, which are
    // zero only once.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(p->stream, &cap);
    if (e != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return fail(GMM_ECUDA, "gmm_pool_tick: a pool's ticks cannot be captured");
    }
    return pool_tick_impl(p, true);
}

int gmm_pool_set_stream(gmm_pool_t *p, void *cuda_stream) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_set_stream: null pool");
    p->stream = static_cast<cudaStream_t>(cuda_stream);
    return GMM_OK;
}

int gmm_pool_set_launch(gmm_pool_t *p, int threads, int ctas_per_sm, int tile_pixels) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_set_launch: null pool");
    const int t = threads ? threads : p->threads;
    const int c = ctas_per_sm ? ctas_per_sm : p->ctas_per_sm;
    // leaving the flat form without a tile size: the default tile
    const int tp = tile_pixels ? tile_pixels : (c >= 0 && p->ctas_per_sm < 0) ? 2048 : p->tile_pixels;
    if (t < 64 || t > 256 || t % 32)
        return fail(GMM_EINVAL, "gmm_pool_set_launch: threads must be 64..256, a multiple of 32");
    if (c < -1 || c > 32)
        return fail(GMM_EINVAL, "gmm_pool_set_launch: ctas_per_sm must be in [-1, 32]");
    if (c >= 0 && (tp < t || tp % t || tp > (1 << 24)))
        return fail(GMM_EINVAL, "gmm_pool_set_launch: tile_pixels must be a multiple of threads");
    p->threads = t;
    p->ctas_per_sm = c;
    p->tile_pixels = tp;
    return GMM_OK;
}

int gmm_pool_set_prefetch(gmm_pool_t *p, int enable) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_set_prefetch: null pool");
    p->prefetch = enable != 0; // picks the kernel instance from the next tick
    return GMM_OK;
}

int gmm_pool_use_graph(gmm_pool_t *p, int enable) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_use_graph: null pool");
    (void)enable; // a tick is one launch per 128 cameras and nothing else
    return GMM_OK;
}

int gmm_pool_autotune_online(gmm_pool_t *p, int ticks_per_shape) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_autotune_online: null pool");
    if (ticks_per_shape < 1 || ticks_per_shape > 1000)
        return fail(GMM_EINVAL, "gmm_pool_autotune_online: ticks_per_shape must be in [1, 1000]");
    DeviceGuard g(p->device);
    const int rc = tuning_poll(p, true); // finish an earlier run first
    if (rc != GMM_OK)
        return rc;
    Tuning &tu = p->tune;
    if (tu.open.a) { // an unfinished run's last trial: no tick will end it now
        cudaEventDestroy(tu.open.a);
        tu.open = Trial();
    }
    tu.cands = tuning_candidates(p);
    tu.ms.assign(tu.cands.size(), {});
    tu.per_shape = ticks_per_shape;
    tu.issued = 0;
    tu.final_round = false;
    tu.named = false;
    tu.active = true;
    return GMM_OK;
}

int gmm_pool_tuning(gmm_pool_t *p, int *threads, int *ctas_per_sm, int *tile_pixels) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_tuning: null pool");
    DeviceGuard g(p->device);
    const int rc = tuning_poll(p, false);
    if (rc != GMM_OK)
        return rc;
    if (threads)
        *threads = p->threads;
    if (ctas_per_sm)
        *ctas_per_sm = p->ctas_per_sm;
    if (tile_pixels)
        *tile_pixels = p->tile_pixels;
    return p->tune.active ? 1 : 0;
}

int gmm_pool_autotune(gmm_pool_t *p, int iters, int *threads_out, int *ctas_out,
                      int *tile_out) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_autotune: null pool");
    if (iters < 1)
        return fail(GMM_EINVAL, "gmm_pool_autotune: iters must be >= 1");
    if (p->sticky != cudaSuccess)
        return fail(GMM_ECUDA, "gmm_pool_autotune: earlier CUDA failure");
    bool any = false;
    size_t snap_bytes = 0;
    for (const PoolCam &c : p->cams)
        if (c.used && c.submitted) {
            any = true;
            snap_bytes += c.L.total;
        }
    if (!any)
        return fail(GMM_EINVAL, "gmm_pool_autotune: no camera has a submitted frame");
    DeviceGuard g(p->device);
    // Snapshot every submitted camera's state so the trials leave no trace.
    uint8_t *snap = nullptr;
    cudaError_t e = cudaMalloc(&snap, snap_bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(GMM_ENOMEM, "gmm_pool_autotune: no room for the state snapshot");
    }
    std::vector<int> init_saved(p->cams.size());
    size_t off = 0;
    e = order_before(p);
    for (size_t i = 0; i < p->cams.size() && e == cudaSuccess; ++i) {
        PoolCam &c = p->cams[i];
        init_saved[i] = c.initialized;
        if (c.used && c.submitted) {
            e = cudaMemcpyAsync(snap + off, c.arena, c.L.total, cudaMemcpyDeviceToDevice, p->stream);
            off += c.L.total;
        }
    }
    cudaEvent_t t0 = nullptr, t1 = nullptr;
    if (e == cudaSuccess)
        e = cudaEventCreate(&t0);
    if (e == cudaSuccess)
        e = cudaEventCreate(&t1);
    const int saved_t = p->threads, saved_c = p->ctas_per_sm, saved_tp = p->tile_pixels;
    int best_t = saved_t, best_c = saved_c, best_tp = saved_tp;
    float best_ms = -1.f;
    const std::vector<Shape> cands =
        distinct_shapes(tuning_candidates(p), submitted_cams(p),
                        [&](const Shape &s) { return blocks_for(p, s.threads, s.ctas); });
    int rc = GMM_OK;
    // Two passes over the candidates (the best time of each counts), so a
    // transient slowdown during one trial does not decide the shape.
    for (int pass = 0; pass < 2; ++pass) {
        for (const Shape &sh : cands) {
            if (e != cudaSuccess || rc != GMM_OK)
                break;
            p->threads = sh.threads;
            p->ctas_per_sm = sh.ctas;
            p->tile_pixels = sh.tile;
            rc = pool_tick_impl(p, false); // warm-up of this shape
            if (rc != GMM_OK)
                break;
            e = cudaEventRecord(t0, p->stream);
            for (int k = 0; k < iters && rc == GMM_OK; ++k)
                rc = pool_tick_impl(p, false);
            if (e == cudaSuccess)
                e = cudaEventRecord(t1, p->stream);
            if (e == cudaSuccess)
                e = cudaEventSynchronize(t1);
            float ms = 0.f;
            if (e == cudaSuccess)
                e = cudaEventElapsedTime(&ms, t0, t1);
            if (e == cudaSuccess && rc == GMM_OK && (best_ms < 0.f || ms < best_ms)) {
                best_ms = ms;
                best_t = sh.threads;
                best_c = sh.ctas;
                best_tp = sh.tile;
            }
            for (PoolCam &cam : p->cams)
                if (cam.used && cam.submitted)
                    cam.initialized = 1; // later trials update, as real ticks would
        }
    }
    // Restore the snapshot and the initialisation flags.
    off = 0;
    for (size_t i = 0; i < p->cams.size(); ++i) {
        PoolCam &c = p->cams[i];
        c.initialized = init_saved[i];
        if (c.used && c.submitted) {
            const cudaError_t er = cudaMemcpyAsync(c.arena, snap + off, c.L.total,
                                                   cudaMemcpyDeviceToDevice, p->stream);
            if (e == cudaSuccess)
                e = er;
            off += c.L.total;
        }
    }
    const cudaError_t es = cudaStreamSynchronize(p->stream);
    if (e == cudaSuccess)
        e = es;
    cudaFree(snap);
    if (t0)
        cudaEventDestroy(t0);
    if (t1)
        cudaEventDestroy(t1);
    if (e != cudaSuccess)
        return cuda_fail(&p->sticky, e, "gmm_pool_autotune");
    if (rc != GMM_OK)
        return rc;
    p->threads = best_t;
    p->ctas_per_sm = best_c;
    p->tile_pixels = best_tp;
    if (threads_out)
        *threads_out = best_t;
    if (ctas_out)
        *ctas_out = best_c;
    if (tile_out)
        *tile_out = best_tp;
    return GMM_OK;
}

int gmm_pool_state_get(const gmm_pool_t *p, int cam, int plane, int component,
                       float *dst_host, size_t n) {
    if (!valid_cam(p, cam))
        return fail(GMM_EINVAL, "gmm_pool_state_get: unknown camera");
    DeviceGuard g(p->device);
    gmm_pool *pm = const_cast<gmm_pool *>(p);
    const PoolCam &c = p->cams[cam];
    const cudaError_t e = order_before(pm);
    if (e != cudaSuccess)
        return cuda_fail(&pm->sticky, e, "gmm_pool_state_get");
    return state_get_common(c.cfg, c.L, c.arena, p->stream, &pm->sticky, plane, component,
                            dst_host, n);
}

size_t gmm_pool_state_used(const gmm_pool_t *p) { return p ? p->used_bytes : 0; }

int gmm_pool_sync(gmm_pool_t *p) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_sync: null pool");
    DeviceGuard g(p->device);
    cudaError_t e = cudaStreamSynchronize(p->stream);
    if (e == cudaSuccess)
        e = wait_for_work(p); // it may have gone to an earlier stream
    if (e != cudaSuccess)
        return cuda_fail(&p->sticky, e, "gmm_pool_sync");
    return p->sticky == cudaSuccess ? GMM_OK : fail(GMM_ECUDA, "gmm_pool_sync: earlier CUDA failure");
}

int gmm_pool_destroy(gmm_pool_t *p) {
    if (!p)
        return fail(GMM_EINVAL, "gmm_pool_destroy: null pool");
    DeviceGuard g(p->device);
    cudaStreamSynchronize(p->stream);
    wait_for_work(p);
    for (Trial &tr : p->tune.pending) {
        cudaEventDestroy(tr.a);
        cudaEventDestroy(tr.b);
    }
    p->tune.pending.clear();
    if (p->tune.open.a)
        cudaEventDestroy(p->tune.open.a);
    p->tune.open = Trial();
    for (PoolCam &c : p->cams)
        if (c.used && c.arena)
            cudaFreeAsync(c.arena, p->stream);
    cudaStreamSynchronize(p->stream);
    if (p->mempool)
        cudaMemPoolDestroy(p->mempool);
    if (p->d_counters)
        cudaFree(p->d_counters);
    if (p->ev_work)
        cudaEventDestroy(p->ev_work);
    delete p;
    return GMM_OK;
}

} // extern "C"
