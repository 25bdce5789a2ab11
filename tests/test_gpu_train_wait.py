"""A wait of the FP32 training convolutions of 16 channels that runs out (forced by
a budget of 0): currents and gradients become NaN, the call returns, and the next
call on the same context equals the one before.  One shape has fewer chunks of 8
steps than resident CTAs, one has several per CTA (which then start within a clip
and in another tile)."""
import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,L,kt,ks0,B,K,H,W", [(1, 5, 7, 3, 1, 12, 20, 24), (0, 3, 9, 0, 3, 33, 64, 64)])
def test_fp32_wait_timeout_leaves_nan_and_recovers(kind, L, kt, ks0, B, K, H, W):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import _lib, api, training as tr
    d = inputs.random_evsnet(kind, L, 16, kt, 1, seed=3, vth=0.2, beta=0.9, std=0.1, ks0=ks0)
    lf = torch.as_tensor(np.stack([inputs.random_logl_clip(3 + b, K + 1, H, W, step_std=0.3) for b in range(B)])).cuda()
    E = torch.as_tensor(np.random.default_rng(9).choice([-1, 0, 0, 1], (B, K, H, W)).astype(np.float32)).cuda()
    meta = api.EvsNetDev.from_dict(d)

    def forward():
        return tr.train_forward(lf, meta, meta.w, meta.b, ckpt_every=8, want_I=True)

    ref = forward()
    _, on, off = tr.emd_count_loss(ref["spikes"], E, 0.01)

    def backward():
        return torch.cat(tr.train_backward(lf, meta, meta.w, meta.b, ref["V_ckpt"], on, off, ckpt_every=8))

    g = backward()
    assert torch.isfinite(ref["I"]).all() and torch.isfinite(g).all() and g.abs().max() > 0
    lib = _lib.load()
    try:
        lib.et_set_wait_budget(0)
        bad_I, bad_g = forward()["I"], backward()
        torch.cuda.synchronize()
        assert torch.isnan(bad_I).all() and torch.isnan(bad_g).any()
    finally:
        lib.et_set_wait_budget(-1)
    assert torch.equal(forward()["I"], ref["I"])
    assert (backward() - g).norm() <= 1e-5 * g.norm()
