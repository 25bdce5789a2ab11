"""The FP32 pixel-wise form at kt = 7 and 13 to 16 channels, whose calls go to one of
two kernels by size: a clip whose calls change from one to the other (single steps
and eight steps of a frame that fills the device; a small frame) equals one call and,
on the small frame, the oracle; the currents agree bit for bit."""
import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,L,C,ks0,H,W", [(1, 3, 16, 0, 360, 640), (1, 3, 13, 5, 361, 639), (0, 2, 14, 7, 187, 253),
                                              (1, 7, 16, 3, 360, 640), (1, 5, 15, 5, 19, 23)])
def test_routes_agree(orc, kind, L, C, ks0, H, W):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import api
    d = inputs.random_evsnet(kind, L, C, 7, 1, seed=L + C, vth=0.3, beta=0.9, std=0.15, ks0=ks0)
    net = api.EvsNetDev.from_dict(d)
    calls = (1, 1, 8, 1, 3, 16)
    lf = inputs.random_logl_clip(W, sum(calls), H, W, step_std=0.4)
    g = torch.as_tensor(lf).cuda()
    whole, steps = api.EvsStateDev(net, H, W), api.EvsStateDev(net, H, W)
    buf, wI, wS = api.evsnet_forward(g, net, whole, want_I=True, want_spikes=True)
    I, S, at, n_ev = [], [], 0, 0
    for n in calls:
        b, i, s = api.evsnet_forward(g[at:at + n].contiguous(), net, steps, t0=at, want_I=True, want_spikes=True)
        I.append(i)
        S.append(s)
        n_ev += b.n()
        at += n
    assert torch.equal(torch.cat(I), wI) and torch.equal(torch.cat(S), wS) and buf.n() == n_ev > 0
    assert torch.equal(steps.V, whole.V) and torch.equal(steps.hist, whole.hist)
    if H * W < 1000:
        onet = orc.EvsNet.from_dict(d)
        oI = orc.evsnet_forward(lf, onet, orc.EvsState.new(onet, H, W), want_I=True)[1]
        assert (np.abs(wI.cpu().numpy() - oI) <= 1e-5 * (1 + np.abs(oI))).all()
