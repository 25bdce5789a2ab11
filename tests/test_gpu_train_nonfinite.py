"""An infinite activation in one channel of one pixel-step makes exactly those
entries of the next layer's weight gradient non-finite that multiply it: the taps
whose output lies inside the clip and the image, not the products with the padding
of a tile or of a chunk of steps.  (The next layer weighs the channel negatively,
so that its own outputs there are zero and everything behind stays finite.)"""
import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import _lib, inputs

pytestmark = pytest.mark.gpu

C, CH = 16, 3                            # channels, the one that overflows


def _nonfinite(dtype, kt, ks, B, K, H, W, at):
    """Whether each entry [co, ci, tap] of layer 1's weight gradient is non-finite, with an
    infinite input in channel CH at (step, row, column) `at` of clip 0."""
    from paper_2508_18071_gb300 import api, training as tr
    d = inputs.random_evsnet(0, 2, C, kt, ks, seed=3, vth=0.3, beta=0.9, std=0.1)
    taps, t0 = kt * ks * ks, kt - 1 if kt > 1 else 4
    w0 = np.zeros((C, taps), np.float32)
    w0[:, t0] = 0.1
    w0[CH, t0] = 2.0
    w1 = d["w"][C * taps:-C].reshape(C, C, taps)
    w1[:, CH] = -0.1
    d["w"] = np.concatenate([w0.ravel(), w1.ravel(), d["w"][-C:]])
    d["b"][:] = 0.05
    s, y, x = at
    lf = inputs.random_logl_clip(1, K + 1, H, W, step_std=0.2)[None].repeat(B, 0)
    lf[0, s + 1, y, x] = 3e38
    meta = api.EvsNetDev.from_dict(d, dtype)
    l = torch.as_tensor(lf).cuda()
    out = tr.train_forward(l, meta, meta.w, meta.b, ckpt_every=8, want_I=True)
    assert torch.isfinite(out["I"]).all()
    on, off = torch.ones_like(l[:, 1:]).contiguous(), torch.zeros_like(l[:, 1:]).contiguous()
    gw, _ = tr.train_backward(l, meta, meta.w, meta.b, out["V_ckpt"], on, off, ckpt_every=8)
    return ~torch.isfinite(gw[C * taps:-C].reshape(C, C, taps)).cpu().numpy()


@pytest.mark.parametrize("dtype", [_lib.ET_F32, _lib.ET_BF16])
@pytest.mark.parametrize("kt,K,step", [(7, 5, 4), (7, 5, 2), (7, 6, 5), (4, 33, 31), (4, 33, 32)])
def test_temporal(dtype, kt, K, step):
    assert torch.cuda.is_available()
    got = _nonfinite(dtype, kt, 1, 2, K, 9, 31, (step, 4, 30))
    want = np.zeros_like(got)
    want[:, CH, [t for t in range(kt) if step + kt - 1 - t < K]] = True
    np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("H,W,y,x", [(20, 48, 5, 47), (20, 48, 0, 0), (17, 50, 16, 49), (9, 64, 8, 31), (8, 33, 7, 32)])
def test_3x3(H, W, y, x):
    assert torch.cuda.is_available()
    got = _nonfinite(_lib.ET_F32, 1, 3, 2, 6, H, W, (2, y, x))
    want = np.zeros_like(got)
    # tap t multiplies the output at the mirrored offset
    want[:, CH, [t for t in range(9) if 0 <= y + 1 - t // 3 < H and 0 <= x + 1 - t % 3 < W]] = True
    np.testing.assert_array_equal(got, want)
