"""gmm_apply_host on a handle that ticks with the staged kernel: page-locked
frames give the masks and the state of device frames."""
import numpy as np
import pytest

import paper_2110_14934_gb300 as G
from parity import scene_frames, to_dev, words

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,M,prec", [(16, 256, 3, G.PREC_F32), (33, 96, 5, G.PREC_F16)])
def test_page_locked_frames_on_the_staged_kernel(H, W, M, prec):
    import torch
    rgb, depth, _ = scene_frames(62, H, W, 1, 44, 5)
    ref, host = G.GMM(H, W, M, precision=prec), G.GMM(H, W, M, precision=prec)
    host.set_kernel(G.KERNEL_STAGED)
    mask = torch.zeros((H, G.mask_words_per_row(W)), dtype=torch.int32).pin_memory()
    for t in range(5):
        want = words(ref.apply(*to_dev(rgb[t], depth[t])))
        r, d = torch.from_numpy(rgb[t]).pin_memory(), torch.from_numpy(depth[t].view(np.int16)).pin_memory()
        got = host.apply_host(r.numpy(), d.numpy(), mask.numpy().view(np.uint32))
        assert np.array_equal(got, want), t
    host.sync()
    assert np.array_equal(host.planes(), ref.planes())
    assert np.array_equal(host.fusion(), ref.fusion())
