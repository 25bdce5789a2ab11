"""FP32 pixel-wise form at kt = 7 and 13 to 16 channels (history in shared memory):
step counts around the chunk's 2, 4 and 8, states carried across calls, ragged
32-pixel tiles, one and several layers (the last layer's output has slots of its
own below four layers), stem and temporal layer 0.  Currents and carried history
within 1e-5 (1 + |value|) of the oracle's, as in test_gpu_events; one call equals
the same steps in several calls bit for bit."""
import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import inputs

pytestmark = pytest.mark.gpu

CALLS = (3, 1, 2, 4, 5, 8, 9, 7)     # frames per call; the first sets the state


@pytest.mark.parametrize("kind,L,C,ks0,H,W", [(0, 2, 16, 0, 5, 13), (1, 3, 14, 3, 3, 11), (0, 4, 13, 5, 1, 33),
                                              (1, 7, 16, 0, 8, 16), (1, 7, 16, 3, 9, 71)])
def test_pix16(orc, kind, L, C, ks0, H, W):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import api
    d = inputs.random_evsnet(kind, L, C, 7, 1, seed=L + C, vth=0.3, beta=0.9, std=0.15, ks0=ks0)
    lf = inputs.random_logl_clip(W, sum(CALLS), H, W, step_std=0.4)
    onet = orc.EvsNet.from_dict(d)
    ost = orc.EvsState.new(onet, H, W)
    net = api.EvsNetDev.from_dict(d)
    st, whole = api.EvsStateDev(net, H, W), api.EvsStateDev(net, H, W)
    oI = orc.evsnet_forward(lf, onet, ost, want_I=True)[1]
    I, S, at, n_ev = [], [], 0, 0
    for n in CALLS:
        part = torch.as_tensor(lf[at:at + n].copy()).cuda()
        buf, i, s = api.evsnet_forward(part, net, st, t0=at, want_I=True, want_spikes=True)
        I.append(i)
        S.append(s)
        n_ev += buf.n()
        at += n
    I, S = torch.cat(I), torch.cat(S)
    gI = I.cpu().numpy()
    assert (np.abs(gI - oI) <= 1e-5 * (1 + np.abs(oI))).all()
    assert n_ev == int((S != 0).sum().item()) > 0
    buf, wI, wS = api.evsnet_forward(torch.as_tensor(lf).cuda(), net, whole, want_I=True, want_spikes=True)
    assert torch.equal(wI, I) and torch.equal(wS, S) and buf.n() == n_ev
    assert torch.equal(whole.V, st.V) and torch.equal(whole.hist, st.hist)
    oh = np.asarray(ost.hist, np.float64).reshape(-1)
    gh = st.hist.cpu().numpy().astype(np.float64)
    assert (np.abs(gh - oh) <= 1e-5 * (1 + np.abs(oh))).all()
