"""One tick from states where neighbouring pixels take every route through the
mixture update: each component matched, a miss, components that change places
(also several at once), depth readings missing, depth models not started. The
direct kernel moves only what a pixel needs and changes, lane by lane, so it
is held against the staged kernel, which moves every pixel's whole state
(bit for bit), and against the oracle (the augmented mode, which has no
staged form)."""
import numpy as np
import pytest

import paper_2110_14934_gb300 as G
from parity import AugPair, Pair, aug_state_mismatch, mask_mismatch, state_mismatch, to_dev, words

pytestmark = pytest.mark.gpu

SHAPES = [(1, 31, 3), (3, 85, 4), (16, 16, 5), (5, 257, 5), (40, 96, 3), (61, 419, 4)]


def _random_case(H, W, M, seed, sort):
    """Planes, List-1 bytes and a frame. sort: components in rank order, as a
    tick leaves them; else in any order (a state loaded by a caller). The
    colour and depth samples lie on a random component or anywhere."""
    rng = np.random.default_rng(seed)
    planes = np.zeros((M, 8, H, W), np.float32)
    for w0, v0, mus, top in ((G.PLANE_W_C, G.PLANE_V_C, (1, 2, 3), 255.0),
                             (G.PLANE_W_D, G.PLANE_V_D, (6,), 4000.0)):
        w = rng.uniform(0.01, 1.0, (M, H, W)) ** 3
        w = w / w.sum(0)
        v = rng.uniform(1.0, 300.0, (M, H, W))
        if sort:
            order = np.argsort(-w / np.sqrt(v), axis=0, kind="stable")
            w, v = np.take_along_axis(w, order, 0), np.take_along_axis(v, order, 0)
        planes[:, w0], planes[:, v0] = w, v
        for m in mus:
            planes[:, m] = rng.uniform(0.0, top, (M, H, W))
    pick = rng.integers(0, M + 1, (H, W))  # M: anywhere
    at = np.minimum(pick, M - 1)[None, None]
    mean = np.take_along_axis(planes, np.broadcast_to(at, (1, 8, H, W)), 0)[0]
    rgb = np.where((pick < M)[None], mean[1:4], rng.uniform(0, 255, (3, H, W)))
    rgb = np.rint(np.moveaxis(rgb, 0, 2)).astype(np.uint8)
    pick_d = rng.integers(0, M + 1, (H, W))
    mean_d = np.take_along_axis(planes[:, 6], np.minimum(pick_d, M - 1)[None], 0)[0]
    depth = np.where(pick_d < M, mean_d, rng.uniform(1, 4000, (H, W)))
    depth = np.maximum(np.rint(depth), 1).astype(np.uint16)
    depth[rng.random((H, W)) < 0.15] = 0
    started = rng.random((H, W)) < 0.85
    count = rng.integers(0, 7, (H, W))
    fusion = rng.integers(0, 2, (H, W)) | (count << 1) | (started.astype(np.int64) << 4)
    planes[:, 5:] *= started
    return planes, fusion.astype(np.uint8), rgb, depth


def _tick(g, rgb, depth):
    import torch
    masks = [g.new_mask() for _ in range(3)]
    g.apply(*to_dev(rgb, depth), *masks)
    torch.cuda.synchronize()
    return [words(m) for m in masks]


@pytest.mark.parametrize("prec", [G.PREC_F32, G.PREC_F16])
@pytest.mark.parametrize("flags", [0, G.FLAG_RHO_ETA | G.FLAG_VAR_PER_CHANNEL])
@pytest.mark.parametrize("sort", [True, False])
@pytest.mark.parametrize("H,W,M", SHAPES)
def test_direct_equals_staged_on_every_route(H, W, M, sort, flags, prec):
    planes, fusion, rgb, depth = _random_case(H, W, M, 17 * H + W, sort)
    pair = []
    for kernel in (G.KERNEL_DIRECT, G.KERNEL_STAGED):
        g = G.GMM(H, W, M, precision=prec, flags=flags)
        g.set_kernel(kernel)
        g.load_state(planes, fusion)
        masks = [_tick(g, rgb, depth) for _ in range(3)]
        g.sync()
        pair.append((masks, g.planes(), g.fusion()))
    for a, b in zip(pair[0][0], pair[1][0]):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
    assert np.array_equal(pair[0][1], pair[1][1])
    assert np.array_equal(pair[0][2], pair[1][2])


@pytest.mark.parametrize("H,W,M", SHAPES)
def test_every_route_matches_the_oracle(H, W, M):
    planes, fusion, rgb, depth = _random_case(H, W, M, 91 * H + W, True)
    pair = Pair(H, W, M)
    pair.gpu.load_state(planes, fusion)
    pair.sync_oracle_to_gpu()
    g, o = pair.tick(rgb, depth)
    exempt = o["near"] != 0
    mm = mask_mismatch(g, o, exempt)
    assert mm["fused"] == 0 and mm["fg_rgb"] == 0 and mm["fg_d"] == 0, mm
    st = state_mismatch(pair.gpu.planes(), pair.orc.planes(), pair.orc.fusion_bytes(), exclude=exempt)
    assert sum(st["bad"]) == 0, st
    assert np.array_equal(pair.gpu.fusion()[~exempt], pair.orc.fusion_bytes()[~exempt])


@pytest.mark.parametrize("flags", [0, G.FLAG_RHO_ETA])
@pytest.mark.parametrize("H,W,M", SHAPES)
def test_every_augmented_route_matches_the_oracle(H, W, M, flags):
    planes, fusion, rgb, depth = _random_case(H, W, M, 7 * H + W, True)
    planes[:, 5] = 0.0
    planes[:, 7] = 0.0
    planes[:, 6] *= 255.0 / 4095.0
    pair = AugPair(H, W, M, flags=flags)
    pair.gpu.load_state(planes, fusion & 1)
    pair.sync_oracle_to_gpu()
    g, o = pair.tick(rgb, depth)
    exempt = o["near"] != 0
    for k in ("fused", "fg_rgb", "fg_d"):
        assert np.array_equal(g[k][~exempt], o["fg"].astype(bool)[~exempt]), k
    st = aug_state_mismatch(pair.gpu.planes(), pair.orc.planes(), exclude=exempt)
    assert sum(st["bad"].values()) == 0, st
