"""Temporal training at sizes where the split of the work can go wrong: more
chunks of two steps than resident blocks (a block then changes tiles and starts
in the middle of a clip), an odd last step, ragged last tiles, and layer 0's
walks along time and rows beyond one segment.  Short dyadic data as in
test_gpu_train_tct: the BF16 forward equals the FP32 one bit for bit, the FP32
gradients are within 1e-4 of the oracle's, the BF16 ones within (L + 1) u."""
import numpy as np
import pytest
import torch

from test_gpu_train_tct import U_BF16, _dyadic_clips, _dyadic_net, _fwd_bwd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tr():
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import training
    return training


@pytest.mark.parametrize("kind,L,C,kt,ks0,B,K,H,W", [
    (1, 3, 16, 7, 3, 2, 35, 37, 19),     # stem, two row strips, ragged everything
    (1, 3, 16, 7, 0, 2, 67, 33, 40),     # paper form, three walks along time
    (0, 3, 16, 4, 0, 4, 33, 64, 64),     # 2176 chunks on 304 blocks, even kt
    (0, 2, 12, 6, 3, 1, 17, 33, 9),      # fewer than 16 channels
    (0, 2, 16, 1, 3, 1, 5, 3, 130),      # no memory, one pixel row past a tile
])
def test_split_of_the_work(tr, orc, kind, L, C, kt, ks0, B, K, H, W):
    from paper_2508_18071_gb300 import _lib
    d = _dyadic_net(kind, L, C, kt, ks0, seed=5 + K, dens=0.1)
    lf = _dyadic_clips(K, B, K, H, W)
    E = np.random.default_rng(9).choice([-1, 0, 0, 0, 1], (B, K, H, W)).astype(np.float32)
    o32, _, g32 = _fwd_bwd(tr, d, lf, E, _lib.ET_F32, 16)
    o16, _, g16 = _fwd_bwd(tr, d, lf, E, _lib.ET_BF16, 16)
    assert (o32["spikes"] != 0).sum().item() > 20
    for k in ("spikes", "V_ckpt", "I"):
        np.testing.assert_array_equal(o16[k].cpu().numpy(), o32[k].cpu().numpy())
    X = np.diff(lf.astype(np.float64), axis=1)
    _, rgw, rgb = orc.torch_grads(X, E, orc.EvsNet.from_dict(d), smooth=False, alpha=2.0, lam=0.01)
    r = np.concatenate([rgw, rgb])
    assert np.abs(g32 - r).max() <= 1e-4 * np.abs(r).max()
    assert np.linalg.norm(g32 - r) <= 1e-4 * np.linalg.norm(r)
    assert np.linalg.norm(g16 - r) <= (L + 1) * U_BF16 * np.linalg.norm(r)
