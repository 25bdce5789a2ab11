"""The pixel-wise tensor-core form on images of more than two tiles of 128 pixels per
SM: a CTA walks tiles, so every tile after a CTA's first must start from its own
history, input buffers and barrier phases.  Pixels reach at most two rows up or down
(the widest stem here), so currents, spikes, membranes, histories and events of the
whole image equal, bit for bit, those of bands of 64 rows with two rows of margin,
which are small enough that no CTA has a second tile."""
import numpy as np
import pytest
import torch

from paper_2508_18071_gb300 import inputs
from test_gpu_evsnet_tct_fp8 import _calibrate, _run, _sorted

pytestmark = pytest.mark.gpu

BAND, M = 64, 2
CHUNKS = [(0, 3), (3, 4), (4, 9)]          # odd step counts, a call of one step


@pytest.mark.parametrize("dtype", ["ET_BF16", "ET_FP8"])
@pytest.mark.parametrize("form,H,W", [((1, 7, 16, 7, 0), 190, 213),     # ragged last tile, 32-bit history rows
                                      ((1, 7, 16, 7, 0), 161, 244),     # 16-byte history rows, ragged last tile
                                      ((1, 7, 16, 7, 3), 190, 213),     # stem by thread loads
                                      ((1, 7, 16, 7, 3), 161, 256),     # stem by TMA
                                      ((0, 3, 9, 5, 3), 190, 256),      # C 9: half-empty second plane
                                      ((1, 5, 16, 4, 5), 190, 213)])    # the general form, an odd slot pair
def test_tiles_equal_bands(form, H, W, dtype):
    assert torch.cuda.is_available()
    from paper_2508_18071_gb300 import _lib, api
    kind, L, C, kt, ks0 = form
    dt = getattr(_lib, dtype)
    assert H * W > 2 * 152 * 128 and (BAND + 2 * M) * W <= 148 * 128
    d = inputs.random_evsnet(kind, L, C, kt, 1, seed=12, std=0.15, vth=0.1, beta=0.95, ks0=ks0)
    lf = inputs.random_logl_clip(5, 9, H, W, step_std=0.3)
    scales = [0.5] * (L - 1) if dtype == "ET_FP8" else None
    ev, I, S, V, h = _run(api, d, lf, dt, scales, CHUNKS)
    assert len(ev) > 1000
    V, h, seen = V.reshape(H, W), h.reshape(-1, H, W), []
    for y in range(0, H, BAND):
        n = min(BAND, H - y)
        a, b = max(0, y - M), min(H, y + n + M)
        evb, Ib, Sb, Vb, hb = _run(api, d, np.ascontiguousarray(lf[:, a:b]), dt, scales, CHUNKS)
        Vb, hb = Vb.reshape(b - a, W), hb.reshape(-1, b - a, W)
        r = slice(y - a, y - a + n)
        np.testing.assert_array_equal(I[:, y:y + n], Ib[:, r])
        np.testing.assert_array_equal(S[:, y:y + n], Sb[:, r])
        np.testing.assert_array_equal(V[y:y + n], Vb[r])
        np.testing.assert_array_equal(h[:, y:y + n], hb[:, r])
        evb = np.asarray(evb).reshape(-1, 4).copy()
        evb[:, 1] += a
        seen.append(evb[(evb[:, 1] >= y) & (evb[:, 1] < y + n)])
    assert np.array_equal(_sorted(ev), _sorted(np.concatenate(seen)))


def test_calibration_over_tiles():
    """The calibrated scales of an image are the largest of its bands' scales."""
    from paper_2508_18071_gb300 import api
    H, W = 190, 213
    d = inputs.random_evsnet(1, 7, 16, 7, 1, seed=12, std=0.15, vth=0.1, beta=0.95, ks0=0)
    lf = inputs.random_logl_clip(5, 9, H, W, step_std=0.3)
    lf[:, 188] *= 8.0                      # the largest inputs are in a last tile
    bands = [_calibrate(api, d, np.ascontiguousarray(lf[:, y:y + BAND])) for y in range(0, H, BAND)]
    got = _calibrate(api, d, lf)
    np.testing.assert_array_equal(got, np.max(bands, axis=0))
    assert (got > bands[0]).any()
