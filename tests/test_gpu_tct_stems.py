"""Stems of 1, 5 and 7 in the BF16 pixel-wise form: images narrower than the stem and
wider than a tile, calls of odd and even step counts.  The data of test_gpu_evsnet_tct
(every tensor-core operand exact in BF16, checked first): bit-identical to the FP32
path."""
import numpy as np
import pytest
import torch

from test_gpu_evsnet_tct import _dyadic_clip, _dyadic_net, _layer_inputs, _run, _sorted

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,H,W,dens", [((1, 5, 16, 7, 7), 9, 40, 0.02), ((1, 3, 16, 7, 7), 6, 4, 0.03),
                                           ((0, 3, 16, 5, 1), 11, 13, 0.1), ((1, 5, 16, 4, 5), 4, 300, 0.03)])
def test_stems_exact_on_dyadic_data(orc, form, H, W, dens):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import _lib, api
    d = _dyadic_net(*form, seed=4, dens=dens)
    lf = _dyadic_clip(104, 14, H, W)
    X = torch.tensor(np.diff(lf.astype(np.float64), axis=0)[None])
    acts = _layer_inputs(orc, orc.EvsNet.from_dict(d), X)
    assert all(torch.equal(a, a.to(torch.bfloat16).double()) for a in acts)   # precondition
    chunks = [(0, 2), (2, 3), (3, 6), (6, 14)]
    ev32, I32, S32, V32, h32 = _run(api, d, lf, _lib.ET_F32, chunks)
    ev16, I16, S16, V16, h16 = _run(api, d, lf, _lib.ET_BF16, chunks)
    assert np.abs(I32).max() > 0.5 and len(ev32) > 20
    np.testing.assert_array_equal(I16, I32)
    np.testing.assert_array_equal(S16, S32)
    np.testing.assert_array_equal(V16, V32)
    np.testing.assert_array_equal(h16, h32)
    assert np.array_equal(_sorted(ev16), _sorted(ev32))
