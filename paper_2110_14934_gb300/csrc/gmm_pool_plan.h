// How a pool's tick is cut into launches and tiles, and which launch shapes its
// tuner tries. (Plain C++: no CUDA call.)
#pragma once

#include <stdint.h>

#include <algorithm>
#include <vector>

namespace gmmlib {

constexpr int kLaunchCams = 128; // cameras per launch: what its parameters hold

// ctas < 0: the flat (non-persistent) form; tile is then its chunk size.
struct Shape {
    int threads, ctas, tile;
    bool operator==(const Shape &o) const {
        return threads == o.threads && ctas == o.ctas && tile == o.tile;
    }
};

// A camera of the tick: its M and padded pixels, and its slot.
struct TickCam {
    int slot, M;
    int64_t n_pad;
};

// One launch: cameras [first, first + count) of the tick's list, cut into
// tiles of `unit` pixels; m: the M they share (flat form), else 0.
struct LaunchPlan {
    int first, count, m, unit;
};

// Tile size of a launch of the persistent form: the shape's, or less where that
// would leave too few tiles or an uneven last wave. share: a CTA's share of the
// launch's pixels. Large launches: a sixteenth of it, so the CTAs end together.
// Smaller ones: about four pixels per thread, in as many equal parts as the
// share holds. A multiple of the block size. (us per tick, tiles of 256, 512,
// 896, 2048 pixels: 40 cameras of odd sizes, 29 M pixels, FP16/BF16 477, 442,
// 429, 427, and 1280 426; 24 cameras, 17 M pixels, FP16/BF16 332, 311, 304, 308,
// FP32 452, 434, 435, 449; 9 cameras, 6.8 M pixels, FP16/BF16 134, 126, 125,
// 128; 4 cameras, 3.4 M pixels, FP32 102, 103, 107, 119.)
inline int launch_tile(const Shape &s, int64_t pixels, int blocks) {
    const int64_t threads = s.threads, four = 4 * threads;
    const int64_t share = (pixels + blocks - 1) / blocks;
    int64_t tile = share / 16 / threads * threads;
    if (tile < four) {
        const int64_t parts = (share + four - 1) / four;
        tile = ((share + parts - 1) / parts + threads - 1) / threads * threads;
    }
    return tile < s.tile ? (int)tile : s.tile;
}

// The tick's launches over `cams`, which are in order of M: up to kLaunchCams
// cameras each, in the flat form of one M each (a kernel per M).
inline void plan_launches(const std::vector<TickCam> &cams, const Shape &s, int blocks,
                          std::vector<LaunchPlan> &out) {
    const bool flat = s.ctas < 0;
    out.clear();
    for (size_t first = 0, end; first < cams.size(); first = end) {
        int64_t pixels = 0;
        for (end = first; end < cams.size() && end < first + kLaunchCams &&
                          !(flat && cams[end].M != cams[first].M); ++end)
            pixels += cams[end].n_pad;
        out.push_back({(int)first, (int)(end - first), flat ? cams[first].M : 0,
                       flat ? s.tile : launch_tile(s, pixels, blocks)});
    }
}

// The persistent shapes of `shapes` as a tick over `cams` runs them, each once:
// where launch_tile takes smaller tiles than a shape names, the shape is the
// one of those tiles. blocks_of(shape): its CTAs.
template <class BlocksOf>
std::vector<Shape> distinct_shapes(const std::vector<Shape> &shapes,
                                   const std::vector<TickCam> &cams, BlocksOf blocks_of) {
    std::vector<Shape> out;
    std::vector<LaunchPlan> plan;
    for (Shape s : shapes) {
        plan_launches(cams, s, blocks_of(s), plan);
        int tile = 0;
        for (const LaunchPlan &l : plan)
            tile = std::max(tile, l.unit);
        if (tile)
            s.tile = tile;
        if (std::find(out.begin(), out.end(), s) == out.end())
            out.push_back(s);
    }
    return out;
}

} // namespace gmmlib
