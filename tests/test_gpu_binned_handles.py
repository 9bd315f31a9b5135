"""Several binned models alive at once: what one needs of the device does not
depend on the others."""
import numpy as np
import pytest
import torch

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _one_bin(scale=3.0):
    return {"n_bins": 1, "bin0": [0], "nominal": [np.array([scale])], "constrained": [False, True],
            "modifiers": [(0, 0, 0, 1.0, 1.0, None, None), (0, 1, 1, 0.9, 1.1, None, None)], "n_params": 2}


def _points(m, spec, sets, seed):
    rng = np.random.default_rng(seed)
    th = rng.normal(0.0, 0.3, (sets, m.n_params))
    free = [k for k in range(m.n_params) if not spec["constrained"][k]]
    th[:, free] = rng.uniform(0.8, 1.2, (sets, len(free)))
    return rng.poisson(20.0, (sets, m.n_bins)).astype(np.float64), th


def test_a_smaller_model_leaves_a_larger_ones_launches():
    big_spec, small_spec = W.binned_model(), _one_bin()
    big = api.BinnedModel(big_spec)
    counts, th = _points(big, big_spec, 3, 1)
    want, want_g = big.nll_grad(counts, th)
    nu = torch.zeros(3, big.n_bins, dtype=torch.float64, device="cuda")
    big.expected(torch.tensor(th, device="cuda"), nu)
    for _ in range(2):  # a smaller model comes between, then the larger one is called again
        small = api.BinnedModel(small_spec)
        c, t = _points(small, small_spec, 2, 2)
        assert np.all(np.isfinite(small.nll_grad(c, t)[0]))
        got, got_g = big.nll_grad(counts, th)
        assert np.array_equal(got, want) and np.array_equal(got_g, want_g)
        again = torch.zeros_like(nu)
        big.expected(torch.tensor(th, device="cuda"), again)
        torch.cuda.synchronize()
        assert torch.equal(again, nu) and float(nu.min()) > 0.0
