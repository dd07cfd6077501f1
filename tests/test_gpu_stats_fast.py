"""Ensemble statistics at the edges of the one-pixel-per-thread form (list
lengths change behind n = 40 and 80, the general form takes over behind 128):
against numpy in 64 bits.  The integer sums are exact, so mean and standard
deviation carry a few roundings of 2^-53 (the tests allow 1e-14 of the
pixel's largest magnitude); quantiles are one float rounding of the textbook
formula, as before."""
import numpy as np
import pytest

import oracle
from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _stats(x):
    npix = x.shape[1]
    out = [torch.zeros(npix, dtype=t, device="cuda")
           for t in (torch.float64, torch.float64, torch.float32, torch.float32)]
    with rtm.Context(0) as ctx:
        ctx.ensemble_stats(torch.from_numpy(x).cuda(), *out)
        torch.cuda.synchronize()
    return [o.cpu().numpy() for o in out]


@pytest.mark.parametrize("n", [1, 2, 3, 20, 21, 39, 40, 41, 64, 80, 81, 101, 128, 129])
def test_edges_of_the_fast_form(n):
    npix = 613
    x = inputs.normal(n, n * npix).reshape(n, npix)
    x[:, 0:40] *= 10.0 ** (8 * inputs.normal(n + 1, n * 40).reshape(n, 40))  # spread exponents
    x[:, 40:60] = 1500.0 + 1e-3 * x[:, 40:60]                               # std far below the mean
    x[:, 60:80] *= 1e-42                                                    # subnormal
    x[:, 80] = 0.0
    x[:, 81] = -3.25                                                        # constant
    x[::2, 82] = 0.0
    x = x.clip(-3e38, 3e38).astype(np.float32)
    mean, std, q05, q95 = _stats(x)
    m, sd, a, b = oracle.ensemble_stats(x)
    top = np.abs(x.astype(np.float64)).max(0)
    assert np.all(np.abs(mean - m) <= 1e-14 * top)
    assert np.all(np.abs(std - sd) <= 1e-14 * top + 1e-13 * sd)
    assert std[80] == 0.0 and std[81] == 0.0
    assert np.array_equal(q05, a.astype(np.float32)) and np.array_equal(q95, b.astype(np.float32))


@pytest.mark.parametrize("n", [7, 64, 128])
def test_infinities_and_nan_stay_in_their_pixel(n):
    npix = 900
    x = inputs.normal(n, n * npix).reshape(n, npix).astype(np.float32)
    clean = _stats(x)
    x[n // 2, 100] = np.inf
    x[0, 101] = -np.inf
    x[n - 1, 102] = np.nan
    mean, std, q05, q95 = _stats(x)
    assert mean[100] == np.inf and mean[101] == -np.inf and np.isnan(mean[102])
    assert np.all(np.isnan(std[100:103]))
    others = np.r_[0:100, 103:npix]
    for got, want in zip((mean, std), clean):
        assert np.allclose(got[others], want[others], rtol=1e-13, atol=1e-14)
    for got, want in zip((q05, q95), clean[2:]):
        assert np.array_equal(got[others], want[others])
    col = np.sort(x[:, 100].astype(np.float64))
    lo = int(np.floor(0.05 * (n - 1)))
    want = col[lo] + (0.05 * (n - 1) - lo) * (col[min(lo + 1, n - 1)] - col[lo])
    assert q05[100] == np.float32(want)
