"""BF16 3x3 stacks of at most 16 channels: every tile height the kernel picks (4, 6
and 8 blocks), two to six layers, ragged tiles, calls of one frame.  Dyadic data
whose BF16 roundings are exact (checked on the CPU first), so currents, spikes,
membranes and events equal the FP32 path's bit for bit."""
import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import inputs
from test_gpu_events import _dyadic_clip, _dyadic_net, _run, _sorted

CASES = [(187, 253, 4, 16, 0.1), (500, 700, 4, 16, 0.1), (60, 75, 6, 12, 0.04), (41, 33, 5, 16, 0.05),
         (3, 5, 2, 16, 0.1), (130, 27, 3, 9, 0.1)]


def activations_exact(d, lf):
    """Whether every tensor-core layer's input is a BF16 number."""
    x = torch.tensor(np.diff(lf.astype(np.float64), axis=0))[:, None]
    w, C, off = torch.tensor(d["w"], dtype=torch.float64), d["C"], 0
    for i in range(d["n_layers"]):
        n = C * x.shape[1] * 9
        if i and not torch.equal(x, x.to(torch.bfloat16).double()):
            return False
        x = torch.relu(torch.nn.functional.conv2d(x, w[off:off + n].view(C, -1, 3, 3), padding=1))
        off += n
    return bool(x.abs().max() > 0)


@pytest.mark.parametrize("H,W,L,C,dens", CASES)
def test_inputs_are_exact(H, W, L, C, dens):
    h, w = min(H, 60), min(W, 80)
    assert activations_exact(_dyadic_net(3, L=L, C=C, density=dens), _dyadic_clip(4, 7, H, W)[:, :h, :w])


@pytest.mark.gpu
@pytest.mark.parametrize("H,W,L,C,dens", CASES)
def test_tc16(H, W, L, C, dens):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import _lib, api
    d = _dyadic_net(3, L=L, C=C, density=dens)
    lf = _dyadic_clip(4, 7, H, W)
    ev32, I32, S32, V32 = _run(api, d, lf, _lib.ET_F32)
    for chunks in (None, [(0, 2), (2, 3), (3, 7)]):
        ev16, I16, S16, V16 = _run(api, d, lf, _lib.ET_BF16, chunks)
        np.testing.assert_array_equal(I16, I32)
        np.testing.assert_array_equal(S16, S32)
        np.testing.assert_array_equal(V16, V32)
        assert np.array_equal(_sorted(ev16), _sorted(ev32))
