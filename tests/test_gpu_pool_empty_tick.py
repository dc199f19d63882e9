"""A pooled tick without a submitted frame launches nothing, so it is accepted
on a stream that is being captured, as anywhere."""
import pytest

import paper_2110_14934_gb300 as G

pytestmark = pytest.mark.gpu


def test_empty_tick_during_capture():
    import torch
    p = G.Pool()
    p.admit(8, 40, 3)
    x = torch.zeros(4, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        g.capture_begin()
        try:
            x += 1
            p.tick()
        finally:
            g.capture_end()
    g.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [1.0] * 4
    p.close()
