"""The decay convolution's gradient for an event so far below the resolution's
peak that the unnormalised value is subnormal while the density, on a narrow
range, is an ordinary number: finite, and the derivative of log f."""
import numpy as np
import pytest
from scipy.special import erfcx

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _dlogf(t, tau, mu, sg):
    """d log f / d (tau, mu, sigma) of f = exp(-u^2/2) erfcx(z) / 2."""
    u, s = (t - mu) / sg, sg / tau
    z = (s - u) / np.sqrt(2.0)
    r = (2.0 * z * erfcx(z) - 2.0 / np.sqrt(np.pi)) / erfcx(z)
    du = np.array([0.0, -1.0 / sg, -u / sg])
    ds = np.array([-sg / tau**2, 0.0, 1.0 / tau])
    return -u * du + r * (ds - du) / np.sqrt(2.0)


@pytest.mark.parametrize("unit", [1e-12, 1e-10])
def test_an_event_38_sigma_below(unit):
    b = W._Builder()
    x = b.obs(-45.0 * unit, 10.0 * unit)
    th = np.array([1.5, 0.0, 1.0]) * unit
    lo, hi = np.array([0.1, -1.0, 0.1]) * unit, np.array([9.0, 1.0, 9.0]) * unit
    spec = b.spec(b.pdf("gaussexp", x, *[b.param(n, th[k], lo[k], hi[k]) for k, n in enumerate(("tau", "mu", "sg"))]))
    m = api.Model.from_spec(spec)
    assert "kernel=generic" in m.describe()
    near = np.array([1.0, 2.0]) * unit
    _, g = api.nll_grad(m, api.Data.upload(m, [near]), th)
    norm = (g + sum(_dlogf(t, *th) for t in near)) / 2  # d log I / d theta
    for k in (37.5, 38.0, 38.1):
        nll, got = api.nll_grad(m, api.Data.upload(m, [np.append(near, -k * unit)]), th)
        assert np.isfinite(nll)
        want = g + norm - _dlogf(-k * unit, *th)
        # f has some 1e7 steps of the smallest subnormal left
        assert np.all(np.abs(got - want) <= 1e-5 * (np.abs(want) + 1.0 / unit)), (k, got, want)
