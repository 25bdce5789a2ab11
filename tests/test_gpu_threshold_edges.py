"""The threshold generator decides most steps from an FP32 estimate with an error
bound and the rest in FP64.  Inputs at which the two could part: log values at,
just below and just above whole multiples of C from the reference, large
references, thousands of events per step, C outside the estimate's range, NaN
and infinities; frame counts around the 16 a thread loads at once; more events
than a warp gathers.  Events and FP64 state equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _edge_frames(rng, F, H, W, C, scale):
    """Random walks in whole multiples of C, nudged by a few float32 ulps."""
    k = rng.integers(-3, 4, (F, H, W)).cumsum(0)
    l = (scale + k * np.float64(C)).astype(np.float32)
    nudge = rng.integers(-2, 3, (F, H, W))
    for _ in range(2):
        l = np.where(nudge > 0, np.nextafter(l, np.float32(np.inf)),
                     np.where(nudge < 0, np.nextafter(l, np.float32(-np.inf)), l)).astype(np.float32)
        nudge -= np.sign(nudge)
    return l


@pytest.mark.parametrize("F,C,scale,jump", [(17, 0.2, -1.0, 0.0), (16, 0.25, 0.0, 0.0), (33, 0.2, 300.0, 0.0),
                                            (5, 0.01, -2.0, 90.0), (2, 0.2, -1.0, 0.0), (18, 1e-36, 0.0, 0.0),
                                            (6, 1e-4, 0.0, 12.0)])
def test_threshold_edges(orc, F, C, scale, jump):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import api
    H, W = 9, 61
    rng = np.random.default_rng(F)
    l = _edge_frames(rng, F, H, W, C, scale)
    if jump:
        l += (rng.uniform(size=l.shape) < 0.004) * rng.normal(0, jump, l.shape).astype(np.float32)
    if F == 17:
        l[3, 2, :8] = [np.nan, np.nan, 0, 0, 0, np.nan, 0, 0]
    ref = torch.zeros(H * W, dtype=torch.float64, device="cuda")
    ost = orc.ThresholdState.new(H, W)
    ini = False
    for part in (l[:max(1, F // 2)], l[max(1, F // 2):]):
        t0 = 0 if not ini else max(1, F // 2)
        ev = api.threshold_events(torch.as_tensor(part.copy()).cuda(), C, ref, ini, t0=t0).host()
        oev = orc.threshold_events(part, C, ost, t0=t0)
        np.testing.assert_array_equal(orc.sort_events(ev), orc.sort_events(oev))
        ini = True
    np.testing.assert_array_equal(ref.cpu().numpy(), np.asarray(ost.ref).reshape(-1))
