"""A program's derivative that leaves the finite range at some event spoils its
own parameter's gradient and no other's."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_other_derivatives_stay():
    # f = (p0 + x)^(1/2) exp(-p1 x): at x = 0 and p0 = 1e-310 the value is 1e-155
    # and d log f / d p0 overflows; d log f / d p1 = -x
    b = W._Builder()
    x = b.obs(0.0, 4.0)
    f = b.expr("p0 x + c0 pow x p1 * neg exp *", (0.5,), x, b.param("p0", 1e-310, 0.0, 1.0), b.param("p1", 0.7, 0.0, 5.0))
    m = api.Model.from_spec(b.spec(f))
    th = np.array([1e-310, 0.7])
    _, g = api.nll_grad(m, api.Data.upload(m, [np.array([1.0, 2.0])]), th)
    assert np.all(np.isfinite(g))
    nll, h = api.nll_grad(m, api.Data.upload(m, [np.array([1.0, 2.0, 0.0])]), th)
    assert np.isfinite(nll) and not np.isfinite(h[0])
    norm = (g[1] - 3.0) / 2  # d log I / d p1
    assert abs(h[1] - (g[1] + norm)) <= 1e-12 * (abs(g[1]) + abs(norm))
