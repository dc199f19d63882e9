"""Pooled ticks whose tiles hold several pixels per thread, so that a warp walks
through a tile and moves its next pixels' state ahead: cameras of odd widths
whose last tile ends after some of the steps, in both precisions, with the
prefetch on and off, alone and beside cameras that use the options or the
augmented mode, bit for bit against each camera alone."""
import numpy as np
import pytest

import paper_2110_14934_gb300 as G
from parity import scene_frames, to_dev, words

pytestmark = pytest.mark.gpu

# 475,392 padded pixels: about 3,100 for each of 152 CTAs, tiles of four pixels per thread
CAMS = [(479, 601, 5), (241, 333, 4), (97, 1000, 3)]
OPTIONS = [dict(), dict(flags=G.FLAG_RHO_ETA | G.FLAG_VAR_PER_CHANNEL), dict(mode=G.MODE_AUGMENTED)]
N = 4


@pytest.mark.parametrize("options", [False, True])
@pytest.mark.parametrize("prec", [G.PREC_F32, G.PREC_F16])
@pytest.mark.parametrize("launch", [(64, 1, 2048), (128, 1, 8192)])
def test_several_steps_per_tile_equal_cameras_alone(launch, prec, options):
    import torch
    kw = OPTIONS if options else [dict()] * len(CAMS)
    frames = [[to_dev(r, d) for r, d in zip(*scene_frames(90 + i, H, W, 1, 44, N)[:2])] for i, (H, W, _) in enumerate(CAMS)]
    alone = []
    for (H, W, M), k, f in zip(CAMS, kw, frames):
        g = G.GMM(H, W, M, precision=prec, **k)
        masks = [words(g.apply(r, d)).copy() for r, d in f]
        alone.append((masks, g.planes()))
        g.close()
    for prefetch in (True, False):
        p = G.Pool(precision=prec)
        p.set_launch(*launch)
        p.set_prefetch(prefetch)
        ids = [p.admit(*c, **k) for c, k in zip(CAMS, kw)]
        for t in range(N):
            masks = [torch.empty((H, G.mask_words_per_row(W)), dtype=torch.int32, device="cuda") for H, W, _ in CAMS]
            for i, c in enumerate(ids):
                p.submit(c, *frames[i][t], masks[i])
            p.tick()
            for i, m in enumerate(masks):
                assert np.array_equal(words(m), alone[i][0][t]), (prefetch, t, i)
        for i, c in enumerate(ids):
            assert np.array_equal(p.planes(c), alone[i][1]), (prefetch, i)
        p.close()
