"""The BF16 weight gradient of the temporal form over a batch far larger than the
configured one equals the sum of the clips' gradients: the tensor cores' additions
round towards zero (a relative error of about 2^-26 per addition in a sum of one
sign), so an accumulator's chain must not grow with the batch.  The bar is the
error of a chain of 8 K additions, one tile's K steps."""
import pytest
import torch

from paper_2508_18071_gb300 import _lib, inputs

pytestmark = pytest.mark.gpu


def test_bf16_weight_gradient_of_a_large_batch():
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import api, training as tr
    kt, C, B, K, H, W = 7, 16, 8, 64, 256, 256
    d = inputs.random_evsnet(0, 2, C, kt, 1, seed=3, vth=0.3, beta=0.9, std=0.1)
    d["w"][-C:] = abs(d["w"][-C:])                # one sign throughout
    meta = api.EvsNetDev.from_dict(d, _lib.ET_BF16)
    gen = torch.Generator(device="cuda").manual_seed(1)
    lf = torch.randn((B, K + 1, H, W), generator=gen, device="cuda")
    out = tr.train_forward(lf, meta, meta.w, meta.b, ckpt_every=16, want_S=False)
    on, off = torch.ones_like(lf[:, 1:]).contiguous(), torch.zeros_like(lf[:, 1:]).contiguous()

    def grad(b0, b1):
        gw, _ = tr.train_backward(lf[b0:b1], meta, meta.w, meta.b, out["V_ckpt"][b0:b1].contiguous(), on[b0:b1],
                                  off[b0:b1], ckpt_every=16)
        return gw[C * kt:-C].double()             # the C -> C layer

    whole, parts = grad(0, B), sum(grad(b, b + 1) for b in range(B))
    assert parts.norm() > 0
    assert (whole - parts).norm() <= 8 * K * 2.0 ** -26 * parts.norm()
