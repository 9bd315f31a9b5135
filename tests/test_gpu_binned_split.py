"""The binned pass at the sizes where its kernels split differently: few
datasets (one a thread, samples over several blocks) and many (four a thread,
the last group short), more than one pass takes at once, models without
histosys or without parameters, samples of fewer bins than quarters, and
overlapping samples.  A dataset's NLL and gradient keep their bits whatever
else is in the call; values against the oracle."""
import numpy as np
import pytest

from oracle import binned as B
from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _odd_spec():
    rng = np.random.default_rng(8)
    sizes, starts = [1, 2, 3, 33, 7, 64], [0, 0, 1, 2, 30, 0]
    nominal = [rng.uniform(1, 30, n) for n in sizes]
    nominal[5] = nominal[5] + 20.0
    mods = [(0, 0, 0, 1.0, 1.0, None, None), (5, 0, 0, 1.0, 1.0, None, None)]
    for s in range(6):
        mods += [(s, 1, 1 + (s + j) % 4, 0.9, 1.05 + 0.02 * j, None, None) for j in range(s % 3)]
        mods += [(s, 2, 1 + (s * j) % 4, 1.0, 1.0, nominal[s] * (0.97 - 0.01 * j), nominal[s] * (1.02 + 0.01 * j))
                 for j in range((s * 5) % 7)]
    return {"n_bins": 64, "bin0": starts, "nominal": nominal, "constrained": [False, True, True, True, False],
            "modifiers": mods, "n_params": 5}


def _plain_spec(n_params):
    mods = [(0, 0, 0, 1.0, 1.0, None, None)] if n_params else []
    return {"n_bins": 5, "bin0": [0], "nominal": [np.array([3.0, 4.0, 5.0, 1.0, 0.5])], "constrained": [False] * n_params,
            "modifiers": mods, "n_params": n_params}


SPECS = {"odd": _odd_spec, "no_histosys": lambda: _plain_spec(1), "no_parameters": lambda: _plain_spec(0),
         "workload": lambda: W.binned_model(channels=9, bins=37)}


@pytest.mark.parametrize("name", sorted(SPECS))
def test_bits_and_values(name):
    spec = SPECS[name]()
    om = B.from_spec(spec)
    m = api.BinnedModel(spec)
    P, S = spec["n_params"], 2051  # two passes of at most 1024, and a last one of 3
    rng = np.random.default_rng(3)
    th = rng.normal(0.0, 0.4, (S, P))
    if P:
        th[:, 0] = rng.uniform(0.8, 1.2, S)
    if name == "workload":
        th = W.binned_toy_thetas(S, 4, P)
    base = om.expected(th[0])[0]
    counts = rng.poisson(np.maximum(base, 0.1), (S, len(base))).astype(float)
    nll, g = m.nll_grad(counts, th)
    for t in (0, 1, 1023, 1024, 2047, 2048, 2050):
        ref, rg, scale = om.nll(th[t], counts[t])
        gscale = np.abs(rg).sum() + np.abs(counts[t]).sum() + 1.0
        assert abs(nll[t] - ref) <= 1e-12 * scale, t
        assert np.all(np.abs(g[t] - rg) <= 1e-9 * gscale), t
        n1, g1 = m.nll_grad(counts[t], th[t].reshape(1, P))
        assert n1[0] == nll[t] and np.array_equal(g1[0], g[t]), t
    for k in (2, 5, 130):
        n2, g2 = m.nll_grad(counts[7:7 + k], th[7:7 + k])
        assert np.array_equal(n2, nll[7:7 + k]) and np.array_equal(g2, g[7:7 + k]), k


def test_domain_flag_is_per_dataset_and_reset():
    spec = _plain_spec(1)
    m = api.BinnedModel(spec)
    th = np.ones((1500, 1))
    th[[3, 1203]] = -1.0  # negative rates
    counts = np.full((1500, 5), 2.0)
    nll, _ = m.nll_grad(counts, th, allow_domain=True)
    assert np.array_equal(np.isinf(nll), th[:, 0] < 0)
    nll, _ = m.nll_grad(counts, np.ones((1500, 1)))
    assert np.all(np.isfinite(nll))
