"""Layer 0 of the temporal training forms where its walks along rows or steps are
of different lengths (the longest, one in between, ragged ends), a one-layer
network: short dyadic data, so spikes equal the oracle's exactly; gradients within
1e-4 of the oracle's, the bar of test_gpu_train_temporal."""
import numpy as np
import pytest
import torch

from test_gpu_train_tct import _dyadic_clips, _dyadic_net, _fwd_bwd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,kt,ks0,B,K,H,W", [
    (16, 7, 3, 2, 64, 37, 200), (12, 7, 3, 2, 48, 37, 70), (16, 7, 3, 1, 3, 5, 1),
    (16, 7, 0, 2, 35, 101, 131), (12, 9, 0, 2, 65, 64, 75), (16, 4, 0, 1, 2, 3, 5),
])
def test_walks(orc, C, kt, ks0, B, K, H, W):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import _lib, training as tr
    d = _dyadic_net(0, 1, C, kt, ks0, seed=5 + K, dens=0.1)
    lf = _dyadic_clips(K, B, K, H, W)
    E = np.random.default_rng(9).choice([-1, 0, 0, 0, 1], (B, K, H, W)).astype(np.float32)
    out, _, g = _fwd_bwd(tr, d, lf, E, _lib.ET_F32, 16)
    X = np.diff(lf.astype(np.float64), axis=1)
    net = orc.EvsNet.from_dict(d)
    on, off, _, _ = orc.torch_forward(torch.tensor(X), net)
    np.testing.assert_array_equal(out["spikes"].cpu().numpy(), (on - off).numpy().astype(np.int8))
    assert (out["spikes"] != 0).sum().item() > 2
    _, rgw, rgb = orc.torch_grads(X, E, net, smooth=False, alpha=2.0, lam=0.01)
    r = np.concatenate([rgw, rgb])
    assert np.abs(g - r).max() <= 1e-4 * np.abs(r).max()
    assert np.linalg.norm(g - r) <= 1e-4 * np.linalg.norm(r)
