"""The FP32 pixel-wise form with its history in shared memory on images of more than
two tiles of 32 pixels per SM: a CTA walks tiles, so every tile after its first must
start from its own history, inputs and membranes.  Pixels reach at most one row up or
down (the stem), so currents, spikes, membranes, histories and event counts of the
whole image equal, bit for bit, those of bands of rows of at most one tile per SM."""
import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import inputs

pytestmark = pytest.mark.gpu

CALLS = (3, 1, 2, 9)


def _run(api, net, lf):
    st = api.EvsStateDev(net, lf.shape[1], lf.shape[2])
    I, S, at, n = [], [], 0, 0
    for k in CALLS:
        buf, i, s = api.evsnet_forward(lf[at:at + k].contiguous(), net, st, t0=at, want_I=True, want_spikes=True)
        I.append(i)
        S.append(s)
        n += buf.n()
        at += k
    H, W = st.H, st.W
    return torch.cat(I), torch.cat(S), st.V.view(H, W), st.hist.view(-1, H, W), n


@pytest.mark.parametrize("kind,L,C,ks0", [(1, 7, 16, 0), (1, 7, 16, 3), (0, 3, 13, 3)])
def test_tiles_equal_bands(kind, L, C, ks0):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import api
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    W = 61
    rows = sms * 32 // W - 2                         # a band with its margin: one tile per SM
    H = 2 * rows + 31
    assert H * W > 2 * sms * 32
    d = inputs.random_evsnet(kind, L, C, 7, 1, seed=L + C, vth=0.3, beta=0.9, std=0.15, ks0=ks0)
    net = api.EvsNetDev.from_dict(d)
    lf = torch.as_tensor(inputs.random_logl_clip(5, sum(CALLS), H, W, step_std=0.4)).cuda()
    I, S, V, h, n = _run(api, net, lf)
    assert n == int((S != 0).sum().item()) > 0
    for y in range(0, H, rows):
        m = min(rows, H - y)
        a, b = max(0, y - 1), min(H, y + m + 1)
        bI, bS, bV, bh, _ = _run(api, net, lf[:, a:b])
        r = slice(y - a, y - a + m)
        assert torch.equal(I[:, y:y + m], bI[:, r]) and torch.equal(S[:, y:y + m], bS[:, r])
        assert torch.equal(V[y:y + m], bV[r]) and torch.equal(h[:, y:y + m], bh[:, r])
