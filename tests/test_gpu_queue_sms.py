"""Ray queues around the rays that all resident traversal warps take without an atomic
(12 blocks of 4 warps of 32 rays on each SM of this device): exactly as many, a row
less, a row more.  The path records equal the one-kernel schedule's."""
import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [95, 96, 97])
def test_queue_length_by_sms(H):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import _lib, api
    W = 16 * torch.cuda.get_device_properties(0).multi_processor_count     # 96 W = 12 * 128 rays per SM
    g = api.Scene(inputs.cornell_box())
    rec = []
    for mode in (_lib.ET_RENDER_WAVEFRONT_TILES, _lib.ET_RENDER_MEGAKERNEL):
        g.set_mode(mode)
        rec.append(api.render_frames(g, inputs.cornell_path(1), W, H, 1, 3, 7, records=True)[2].cpu().numpy())
    np.testing.assert_array_equal(rec[0], rec[1])
