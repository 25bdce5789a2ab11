"""Infinite log values count 2^32 - 1 events each (a count saturates) next to the
events of the other pixels of their warp, which reach their own steps at the same
time: the total is exact, the call reports that the buffer is too small, and the
state is the FP64 one."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pixels", [[5], [0, 31, 40], [3, 4]])
def test_infinite_steps(pixels):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import _lib, api
    F, H, W, C = 20, 1, 64, 0.25
    rng = np.random.default_rng(3)
    l = (rng.integers(-3, 4, (F, H, W)) * 0.25).cumsum(0).astype(np.float32)   # exact multiples of C
    for i, p in enumerate(pixels):
        l[7 + 2 * i, 0, p] = np.inf
    ref = torch.zeros(H * W, dtype=torch.float64, device="cuda")
    buf = api.EventBuffer(1 << 12)
    api.threshold_events(torch.as_tensor(l).cuda(), C, ref, False, t0=0, buf=buf)
    r, n = l[0].astype(np.float64).ravel(), 0
    with np.errstate(invalid="ignore"):
        for k in range(1, F):
            d = l[k].astype(np.float64).ravel() - r
            m = np.floor(np.abs(d) / C)
            fire = m > 0
            n += sum(int(min(v, 2.0 ** 32 - 1)) for v in m[fire])
            r[fire] = r[fire] + np.sign(d[fire]) * m[fire] * C
    assert n > len(pixels) * (2 ** 32 - 1)
    assert int(buf.count.item()) == n
    with pytest.raises(_lib.ETError) as e:
        buf.host()
    assert e.value.status == _lib.ET_ERR_CAPACITY
    np.testing.assert_array_equal(ref.cpu().numpy(), r)
