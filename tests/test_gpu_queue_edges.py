"""Ray queues of lengths at which the traversal's fetching can go wrong: fewer
rays than a warp takes, one more than a multiple of 32, exactly the rays that
all resident warps take without an atomic (12 blocks of 4 warps on each of 152
SMs), and one row more.  Every ray must be traced once: the path records equal
the one-kernel schedule's."""
import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(1, 1), (31, 1), (33, 1), (19, 20), (608, 384), (608, 385)])
def test_queue_lengths(W, H):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import _lib, api
    g = api.Scene(inputs.cornell_box())
    out = []
    for mode in (_lib.ET_RENDER_WAVEFRONT_TILES, _lib.ET_RENDER_MEGAKERNEL):
        g.set_mode(mode)
        rgb, _, rec = api.render_frames(g, inputs.cornell_path(1), W, H, 1, 3, 7, records=True)
        out.append((rgb.cpu().numpy(), rec.cpu().numpy()))
    np.testing.assert_array_equal(out[0][1], out[1][1])
    np.testing.assert_allclose(out[0][0], out[1][0], rtol=1e-6, atol=1e-9)
