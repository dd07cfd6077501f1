"""Pixels whose values span more than the integer grid of the fast statistics
holds (2^31 below the largest): their sums are FP64's, in image order, so a
column whose large values cancel keeps the small ones."""
import numpy as np
import pytest

from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _stats(x):
    out = [torch.zeros(x.shape[1], dtype=t, device="cuda")
           for t in (torch.float64, torch.float64, torch.float32, torch.float32)]
    with rtm.Context(0) as ctx:
        ctx.ensemble_stats(torch.from_numpy(x).cuda(), *out)
        torch.cuda.synchronize()
    return [o.cpu().numpy() for o in out]


@pytest.mark.parametrize("n", [3, 40, 41, 64, 81, 128])
def test_small_values_outlive_large_ones_that_cancel(n):
    npix = 300
    x = (1.0 + 0.1 * inputs.normal(n, n * npix).reshape(n, npix)).astype(np.float32)
    wide = np.zeros(npix, bool)
    # powers of two apart: 30 and 31 are on the grid, 32 to 60 are cut, 200 are out of it
    for p, e in enumerate((30, 31, 32, 33, 40, 54, 60, 100, 126)):
        x[0, p], x[1, p] = 2.0 ** e, -(2.0 ** e)
        wide[p] = e >= 33
    x[:, 10] = 0.0
    x[n - 1, 10] = 1e-42          # zeros and one subnormal value: not wide
    x[0, 11], x[1, 11] = 1.0, -1.0
    x[2:, 11] = 1e-42             # subnormal values 2^126 below
    wide[11] = True
    mean, std, _, _ = _stats(x)
    d = x.astype(np.float64)
    s = np.zeros(npix)
    for k in range(n):
        s += d[k]
    m = s / n
    # FP64 in image order, bit for bit
    assert np.array_equal(mean[wide], m[wide])
    # the integer sums are exact: one rounding of the sum, one of the division
    assert np.allclose(mean[~wide], m[~wide], rtol=0, atol=1e-15 * np.abs(d[:, ~wide]).max(0).max())
    assert np.allclose(mean[12:], m[12:], rtol=(n + 2) * 2.0 ** -53, atol=0)  # n roundings of the sum
    sd = np.sqrt(((d - d.mean(0)) ** 2).sum(0) / (n - 1))
    assert np.allclose(std, sd, rtol=1e-13, atol=0)
