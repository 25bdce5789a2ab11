"""The first call on a fresh state with a single frame, as a program makes that
feeds one frame at a time: it has no step, so membrane and history stay exactly
as they were, no event is emitted and the frame becomes the previous one.  The
calls that follow equal one call over the same frames bit for bit (the
pixel-wise BF16 and FP8 forms in pairs of steps, which fix their sum order).
The state starts from short dyadic values, exact in every precision."""
import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import _lib, inputs

pytestmark = pytest.mark.gpu

F32, BF16, FP8 = _lib.ET_F32, _lib.ET_BF16, _lib.ET_FP8


@pytest.mark.parametrize("dtype,kind,L,C,kt,ks,ks0,H,W", [
    # history in shared memory (kt = 7, 13 to 16 channels)
    (F32, 0, 2, 16, 7, 1, 0, 5, 13), (F32, 1, 3, 14, 7, 1, 3, 3, 11), (F32, 0, 4, 13, 7, 1, 5, 1, 33),
    (F32, 1, 7, 16, 7, 1, 0, 8, 16), (F32, 1, 7, 16, 7, 1, 3, 9, 71), (F32, 1, 7, 16, 7, 1, 3, 99, 101),
    # the other pixel-wise and spatial FP32 kernels
    (F32, 1, 3, 8, 5, 1, 0, 9, 15), (F32, 0, 4, 16, 1, 3, 0, 21, 37), (F32, 0, 2, 20, 1, 3, 0, 9, 15),
    # tensor-core forms
    (BF16, 1, 7, 16, 7, 1, 0, 8, 16), (BF16, 1, 7, 16, 7, 1, 3, 9, 71), (BF16, 0, 4, 16, 1, 3, 0, 21, 37),
    (FP8, 1, 7, 16, 7, 1, 3, 9, 71), (FP8, 0, 4, 16, 1, 3, 0, 21, 37)])
def test_first_frame_alone(dtype, kind, L, C, kt, ks, ks0, H, W):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import api
    d = inputs.random_evsnet(kind, L, C, kt, ks, seed=L + C, vth=0.3, beta=0.9, std=0.15, ks0=ks0)
    net = api.EvsNetDev.from_dict(d, dtype)
    if dtype == FP8 and ks == 1:
        net.scales = torch.ones(L - 1, device="cuda")
    K = 8
    lf = torch.as_tensor(inputs.random_logl_clip(W, K + 1, H, W, step_std=0.4)).cuda()
    rng = np.random.default_rng(3)
    steps, whole = api.EvsStateDev(net, H, W), api.EvsStateDev(net, H, W)
    for st in (steps, whole):
        st.last_l.fill_(7.0)
    steps.V.copy_(torch.as_tensor(rng.integers(-2, 3, H * W) / 8.0))
    steps.hist.copy_(torch.as_tensor(rng.integers(0, 8, steps.hist.numel()) / 4.0))
    whole.V.copy_(steps.V)
    whole.hist.copy_(steps.hist)
    V0, hist0 = steps.V.clone(), steps.hist.clone()
    buf, _, _ = api.evsnet_forward(lf[:1].contiguous(), net, steps)
    assert buf.n() == 0 and steps.initialized
    assert torch.equal(steps.V, V0) and torch.equal(steps.hist, hist0)
    assert torch.equal(steps.last_l, lf[0].reshape(-1))
    n = 2 if dtype != F32 and ks == 1 else 1
    I, S, n_ev = [], [], 0
    for k in range(1, K + 1, n):
        buf, i, s = api.evsnet_forward(lf[k:k + n].contiguous(), net, steps, t0=k, want_I=True, want_spikes=True)
        I.append(i)
        S.append(s)
        n_ev += buf.n()
    buf, wI, wS = api.evsnet_forward(lf, net, whole, want_I=True, want_spikes=True)
    assert torch.equal(wI, torch.cat(I)) and torch.equal(wS, torch.cat(S)) and buf.n() == n_ev > 0
    assert torch.equal(whole.V, steps.V) and torch.equal(whole.hist, steps.hist)
