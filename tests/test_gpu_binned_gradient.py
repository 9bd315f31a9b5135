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
