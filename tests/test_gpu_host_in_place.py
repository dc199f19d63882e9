"""gmm_apply_host on page-locked buffers, which the tick reads and writes in
place, against the same frames ticked from device memory: the masks and the
state are the same, also where the buffers rule the direct route out (mask over
the frame, odd alignment, ordinary memory) and between queued frames."""
import numpy as np
import pytest

import paper_2110_14934_gb300 as G
from parity import scene_frames, to_dev, words

pytestmark = pytest.mark.gpu


def _pinned(a):
    import torch
    return torch.from_numpy(a).pin_memory()


@pytest.mark.parametrize("H,W,M,prec,morph", [(1, 1, 3, G.PREC_F32, False), (45, 83, 4, G.PREC_F16, False),
                                              (64, 257, 5, G.PREC_F32, True), (120, 160, 3, G.PREC_F16, True)])
def test_host_frames_in_place_equal_device_frames(H, W, M, prec, morph):
    import torch
    rgb, depth, _ = scene_frames(61, H, W, 1, 44, 8)
    ref, host = (G.GMM(H, W, M, precision=prec, morph_open=morph) for _ in range(2))
    wpr, L = G.mask_words_per_row(W), G.load_library()
    tickets = []
    for t in range(8):
        want = words(ref.apply(*to_dev(rgb[t], depth[t])))
        r, d = _pinned(rgb[t].reshape(-1)), _pinned(depth[t].view(np.int16).reshape(-1))
        m = torch.full((H * wpr + 1,), -1, dtype=torch.int32).pin_memory()
        if t == 5:  # ordinary memory
            got = host.apply_host(rgb[t], depth[t])
        elif t == 6:  # the mask over the start of the colour frame
            buf = torch.zeros(max(3 * H * W, 4 * H * wpr), dtype=torch.uint8).pin_memory()
            buf[:3 * H * W] = r
            assert L.gmm_apply_host(host._h, buf.data_ptr(), d.data_ptr(), buf.data_ptr()) == G.OK
            got = buf[:4 * H * wpr].numpy().view(np.uint32)
        elif t == 7:  # an odd depth address
            buf = torch.zeros(2 * H * W + 1, dtype=torch.uint8).pin_memory()
            buf[1:] = d.view(torch.uint8)
            assert L.gmm_apply_host(host._h, r.data_ptr(), buf.data_ptr() + 1, m.data_ptr()) == G.OK
            got = m[:-1].numpy().view(np.uint32)
        elif t in (2, 3):  # queued, then one that finds a frame in flight
            tickets.append(host.pipe_submit(r, d, m))
            if t == 2:
                host.pipe_wait(tickets[-1])
            else:
                m2 = torch.empty_like(m).pin_memory()
                want = words(ref.apply(*to_dev(rgb[t], depth[t])))
                assert L.gmm_apply_host(host._h, r.data_ptr(), d.data_ptr(), m2.data_ptr()) == G.OK
                host.pipe_wait(tickets[-1])
                m = m2
            got = m[:-1].numpy().view(np.uint32)
        else:
            assert L.gmm_apply_host(host._h, r.data_ptr(), d.data_ptr(), m.data_ptr()) == G.OK
            got = m[:-1].numpy().view(np.uint32)
            assert int(m[-1]) == -1
        assert np.array_equal(np.asarray(got).reshape(H, wpr), want), t
    assert tickets == [2, 3]  # every frame takes a ticket
    assert np.array_equal(host.planes(), ref.planes())
    assert np.array_equal(host.fusion(), ref.fusion())
