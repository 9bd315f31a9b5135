"""Host-buffer calls without the gradient over several sets, on both sides of
the size up to which results come in place (7 doubles a set: 64 KiB lies
between 1170 and 1171): the values of the gradient's call, an empty set, a set
outside the domain."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sets", [3, 1170, 1171])
@pytest.mark.parametrize("which,true", [("decay_model", W.DECAY_TRUE), ("decay_generic_model", W.DECAY_GENERIC_TRUE)])
def test_values_alone(which, true, sets):
    m = api.Model.from_spec(W.model_for(which))
    sizes = np.arange(sets) * 7 % 300 + 5
    sizes[1] = 0
    off = np.concatenate([[0], np.cumsum(sizes)])
    d = api.Data.upload(m, [np.random.default_rng(5).uniform(0.1, 9.0, off[-1])], offsets=off)
    for step in (0.0, 0.01):
        th = np.tile(np.asarray(true) * (1 + step), (sets, 1))
        th[2, 0] = -1.0  # tau < 0
        nll, _ = api.nll_grad(m, d, th, allow_domain=True)
        only = api.nll(m, d, th, allow_domain=True)
        assert only[1] == 0.0 and only[2] == np.inf and nll[2] == np.inf
        good = np.arange(sets) != 2
        assert np.all(np.isfinite(only[good])) and np.allclose(only[good], nll[good], rtol=1e-12, atol=0.0)
        assert np.array_equal(api.nll(m, d, th, allow_domain=True), only)
