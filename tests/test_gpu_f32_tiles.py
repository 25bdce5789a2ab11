"""FP32 3x3 stacks at every depth the tiled kernel takes (two to six layers: 4 to 8
positions of a lane cover a layer's region), ragged tiles, fewer than 16 channels,
calls of one step.  Dyadic data, exact in FP32 whatever the order of the sums, so
currents equal a float64 evaluation bit for bit; events are the spikes."""
import numpy as np
import pytest
import torch

from test_gpu_events import _dyadic_clip, _dyadic_net, _run, _sorted

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,C,H,W,dens", [(2, 16, 16, 32, 0.1), (2, 5, 17, 33, 0.1), (3, 16, 31, 70, 0.1),
                                          (3, 9, 1, 1, 0.1), (4, 16, 50, 97, 0.08), (5, 16, 33, 40, 0.05),
                                          (6, 16, 40, 65, 0.04), (6, 3, 15, 31, 0.2)])
def test_f32_stack(L, C, H, W, dens):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import _lib, api
    d = _dyadic_net(3, L=L, C=C, density=dens)
    lf = _dyadic_clip(4, 7, H, W)
    x = torch.tensor(np.diff(lf.astype(np.float64), axis=0))[:, None]
    w, off = torch.tensor(d["w"], dtype=torch.float64), 0
    for _ in range(L):
        n = C * x.shape[1] * 9
        x = torch.relu(torch.nn.functional.conv2d(x, w[off:off + n].view(C, -1, 3, 3), padding=1))
        assert torch.equal(x, x.float().double())
        off += n
    want = (x * w[off:].view(1, C, 1, 1)).sum(1)
    one = _run(api, d, lf, _lib.ET_F32)
    np.testing.assert_array_equal(one[1], want.numpy())
    ev, S = np.asarray(one[0]).reshape(-1, 4), np.asarray(one[2])
    t, y, x_ = np.nonzero(S)
    assert np.array_equal(_sorted(ev)[:, :2], _sorted(np.stack([x_, y, t, S[t, y, x_]], 1))[:, :2])
    assert len(ev) == np.count_nonzero(S)
    ev2, I2, S2, V2 = _run(api, d, lf, _lib.ET_F32, [(0, 2), (2, 3), (3, 7)])
    np.testing.assert_array_equal(I2, one[1])
    np.testing.assert_array_equal(S2, S)
    np.testing.assert_array_equal(V2, one[3])
    assert np.array_equal(_sorted(ev2), _sorted(ev))
