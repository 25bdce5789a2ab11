"""Training workspaces off 16-byte boundaries: the temporal forms of 16 channels
then take their rows a word at a time.  Currents within 1e-5 (1 + |value|) of the
ones on an aligned workspace (FP32; BF16 rounds the same operands) and gradients
within 1e-4 of their norm (FP32) or (L + 1) 2^-8 (BF16), the bars of the forms'
own tests.  One word off a 4-byte boundary is refused."""
import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import _lib, inputs

pytestmark = pytest.mark.gpu


def _on_workspace(tr, off, fn):
    ws = tr._workspace()
    saved = ws.buf
    ws.buf = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")[off:]
    try:
        assert ws.buf.data_ptr() % 16 == off
        return fn()
    finally:
        ws.buf = saved


@pytest.mark.parametrize("dtype", [_lib.ET_F32, _lib.ET_BF16])
@pytest.mark.parametrize("L,kt,ks0,C", [(1, 7, 0, 16), (1, 7, 3, 16), (1, 9, 0, 16), (1, 5, 5, 16), (3, 7, 0, 16),
                                        (3, 4, 3, 16), (3, 7, 3, 12)])
def test_unaligned_workspace(L, kt, ks0, C, dtype):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import api, training as tr
    if dtype == _lib.ET_BF16 and kt > 7:
        kt = 6
    B, K, H, W = 2, 19, 9, 17
    d = inputs.random_evsnet(1, L, C, kt, 1, seed=3, vth=0.3, beta=0.9, std=0.3, ks0=ks0)
    lf = torch.as_tensor(np.stack([inputs.random_logl_clip(3 + b, K + 1, H, W, step_std=0.3) for b in range(B)])).cuda()
    E = torch.as_tensor(np.random.default_rng(9).choice([-1, 0, 0, 1], (B, K, H, W)).astype(np.float32)).cuda()
    meta = api.EvsNetDev.from_dict(d, dtype)
    ref = tr.train_forward(lf, meta, meta.w, meta.b, ckpt_every=8, want_I=True)
    _, on, off = tr.emd_count_loss(ref["spikes"], E, 0.01)

    def both():
        out = tr.train_forward(lf, meta, meta.w, meta.b, ckpt_every=8, want_I=True)
        return out["I"], torch.cat(tr.train_backward(lf, meta, meta.w, meta.b, ref["V_ckpt"], on, off, ckpt_every=8))

    I, g = both()
    assert g.abs().max() > 0
    tol = 1e-4 if dtype == _lib.ET_F32 else (L + 1) * 2.0 ** -8
    for shift in (4, 8):
        uI, ug = _on_workspace(tr, shift, both)
        assert ((uI - I).abs() <= 1e-5 * (1 + I.abs())).all()
        assert (ug - g).norm() <= tol * g.norm()


def test_workspace_off_a_word_is_refused():
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import api, training as tr
    for kt, ks in ((7, 1), (1, 3)):
        meta = api.EvsNetDev.from_dict(inputs.random_evsnet(0, 2, 16, kt, ks, seed=3))
        lf = torch.zeros((1, 5, 8, 8), device="cuda")
        with pytest.raises(_lib.ETError) as e:
            _on_workspace(tr, 2, lambda: tr.train_forward(lf, meta, meta.w, meta.b, ckpt_every=4))
        assert e.value.status == _lib.ET_ERR_ARG
