"""Pooled ticks on changing streams: each follows the one before it, whatever
stream that ran on, so the models equal those ticked on one stream; and a tick
on a stream that is being captured is refused and changes nothing."""
import numpy as np
import pytest

import paper_2110_14934_gb300 as G
from parity import scene_frames, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [G.PREC_F32, G.PREC_F16])
def test_ticks_follow_one_another_across_streams(prec):
    import torch
    sizes = [(480, 640, 5), (237, 321, 3)]
    frames = [[to_dev(r, d) for r, d in zip(*scene_frames(70 + i, H, W, 1, 44, 12)[:2])] for i, (H, W, _) in enumerate(sizes)]
    streams = [torch.cuda.Stream(), torch.cuda.default_stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    results = []
    for moving in (False, True):
        p = G.Pool(precision=prec)
        cams = [p.admit(*s) for s in sizes]
        # every tick has masks of its own: no tick waits for a reader of another's
        masks = [[torch.zeros((H, G.mask_words_per_row(W)), dtype=torch.int32, device="cuda") for H, W, _ in sizes] for _ in range(12)]
        torch.cuda.synchronize()
        for t in range(12):
            for i, c in enumerate(cams):
                p.submit(c, *frames[i][t], masks[t][i])
            p.tick(stream=streams[t % 3 if moving else 0])
        torch.cuda.synchronize()
        results.append(([m.cpu().numpy() for ms in masks for m in ms], [p.planes(c) for c in cams]))
        p.close()
    (m0, s0), (m1, s1) = results
    assert all(np.array_equal(a, b) for a, b in zip(m0, m1))
    assert all(np.array_equal(a, b) for a, b in zip(s0, s1))


def test_capture_of_a_tick_is_refused():
    import torch
    (rgb, depth, _), (H, W, M) = scene_frames(73, 24, 40, 1, 44, 3), (24, 40, 3)
    p, q = G.Pool(), G.Pool()
    cp, cq = p.admit(H, W, M), q.admit(H, W, M)
    mask = torch.zeros((H, G.mask_words_per_row(W)), dtype=torch.int32, device="cuda")
    s = torch.cuda.Stream()
    for t in range(3):
        r, d = to_dev(rgb[t], depth[t])
        torch.cuda.synchronize()
        for pool, cam in ((p, cp), (q, cq)):
            pool.submit(cam, r, d, mask)
            if pool is p and t == 1:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.stream(s):
                    g.capture_begin()
                    with pytest.raises(G.GMMError):
                        p.tick()
                    g.capture_end()
            pool.tick(stream=s)
            torch.cuda.synchronize()
    assert np.array_equal(p.planes(cp), q.planes(cq))
    p.close()
    q.close()
