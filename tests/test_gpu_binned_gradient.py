"""The binned gradient's terms, each as it is defined."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api

pytestmark = pytest.mark.gpu


def test_a_normfactors_derivative_is_one_rounding_from_its_sum():
    # two normfactors on one sample: with the second one at 1, its derivative is
    # the sample's weighted sum itself, and the first one's that sum over its value
    spec = {"n_bins": 3, "bin0": [0], "nominal": [np.array([3.0, 5.0, 2.5])], "constrained": [False, False],
            "modifiers": [(0, 0, 0, 1.0, 1.0, None, None), (0, 0, 1, 1.0, 1.0, None, None)], "n_params": 2}
    m = api.BinnedModel(spec)
    rng = np.random.default_rng(7)
    th = np.column_stack([rng.uniform(0.3, 3.0, 500), np.ones(500)])
    nll, g = m.nll_grad(rng.poisson(4.0, (500, 3)).astype(np.float64), th)
    assert np.all(np.isfinite(nll)) and np.array_equal(g[:, 0], g[:, 1] / th[:, 0])


def test_a_parameter_with_modifiers_of_every_kind_in_any_order():
    from oracle import binned as B

    h = [np.array([3.0, 5.0, 2.5]), np.array([8.0, 2.0, 4.0, 6.0])]
    ns = lambda s, k: (s, 1, k, 0.9, 1.2, None, None)  # noqa: E731
    nf = lambda s, k: (s, 0, k, 1.0, 1.0, None, None)  # noqa: E731
    hs = lambda s, k: (s, 2, k, 1.0, 1.0, 0.9 * h[s], 1.05 * h[s])  # noqa: E731
    spec = {"n_bins": 5, "bin0": [2, 0], "nominal": h, "constrained": [False, True, False],
            "modifiers": [ns(0, 0), nf(1, 0), hs(1, 0), nf(0, 0), hs(0, 1), ns(1, 1), nf(0, 2), hs(0, 0)], "n_params": 3}
    m, om = api.BinnedModel(spec), B.from_spec(spec)
    rng = np.random.default_rng(9)
    th = np.column_stack([rng.uniform(0.5, 1.8, 200), rng.normal(0.0, 0.5, 200), rng.uniform(0.7, 1.3, 200)])
    counts = rng.poisson(6.0, (200, 5)).astype(np.float64)
    nll, g = m.nll_grad(counts, th)
    for t in range(200):
        ref, rg, scale = om.nll(th[t], counts[t])
        assert abs(nll[t] - ref) <= 1e-12 * scale
        assert np.all(np.abs(g[t] - rg) <= 1e-9 * (np.abs(rg).sum() + counts[t].sum() + 1.0))
