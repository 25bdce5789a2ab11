"""FP32 training of the 3x3 stack at the edges of its tiles (8 rows x 32 columns in
both directions, two rows per warp in the weight gradient): one pixel, exact and
just exceeded tiles, narrow and tall images, fewer than 16 channels, more tiles
than resident blocks.  Bars as in test_gpu_train: spikes equal to the oracle's, whose
potential keeps 1e-5 clear of the thresholds, gradients within 1e-4 of the largest
component and in relative L2."""
import numpy as np
import pytest
import torch

from test_gpu_train import _net, _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,K,H,W,L,C,ck", [(1, 3, 1, 1, 2, 16, 2), (1, 5, 8, 32, 3, 16, 5),
                                            (2, 4, 9, 33, 3, 16, 3), (1, 4, 7, 31, 2, 9, 4),
                                            (1, 6, 3, 70, 2, 3, 4), (1, 3, 70, 2, 3, 13, 3),
                                            (2, 10, 66, 130, 2, 16, 10)])
def test_tile_edges(orc, B, K, H, W, L, C, ck):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import api, training as tr
    d, lf, E = _problem(6, B, K, H, W, L, C)
    onet = _net(orc, d)
    X = np.diff(lf.astype(np.float64), axis=1)
    Son, Soff, oI, Vp = orc.torch_forward(torch.tensor(X), onet)
    assert torch.minimum((Vp - onet.vth).abs(), (Vp + onet.vth).abs()).min().item() > 1e-5
    meta = api.EvsNetDev.from_dict(d)
    lfd = torch.as_tensor(lf).cuda()
    out = tr.train_forward(lfd, meta, meta.w, meta.b, ckpt_every=ck, want_I=True)
    np.testing.assert_allclose(out["I"].cpu().numpy(), oI.numpy(), atol=1e-5 * max(1.0, oI.abs().max().item()))
    np.testing.assert_array_equal(out["spikes"].cpu().numpy(), (Son - Soff).numpy().astype(np.int8))
    _, dSon, dSoff = tr.emd_count_loss(out["spikes"], torch.as_tensor(E).cuda(), 0.01)
    gw, gb = tr.train_backward(lfd, meta, meta.w, meta.b, out["V_ckpt"], dSon, dSoff, ckpt_every=ck)
    _, rgw, rgb = orc.torch_grads(X, E, onet, smooth=False, alpha=2.0, lam=0.01)
    g = np.concatenate([gw.cpu().numpy(), gb.cpu().numpy()]).astype(np.float64)
    r = np.concatenate([rgw, rgb])
    assert np.abs(r).max() > 0
    assert np.abs(g - r).max() <= 1e-4 * np.abs(r).max()
    assert np.linalg.norm(g - r) <= 1e-4 * np.linalg.norm(r)
