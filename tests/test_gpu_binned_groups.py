"""The binned pass with four datasets a thread and a last group of one, two and
three, on the workload model and on samples of fewer bins than quarters,
overlapping and without histosys: a dataset's bits are those of the dataset
alone (one a thread), values against the oracle."""
import numpy as np
import pytest

from oracle import binned as B
from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _odd_samples():
    """360 samples of 1 to 64 bins over the same 64 bins (6600 entries: four a
    thread from 94 datasets on, on 152 SMs)."""
    rng = np.random.default_rng(21)
    sizes, starts = [1, 2, 3, 33, 7, 64] * 60, [0, 0, 1, 2, 30, 0] * 60
    nominal = [rng.uniform(0.1, 1.0, n) for n in sizes]
    mods = [(s, 0, 0, 1.0, 1.0, None, None) for s in range(0, 360, 9)]
    for s in range(360):
        mods += [(s, 1, 1 + (s + j) % 4, 0.9, 1.05 + 0.02 * j, None, None) for j in range(s % 3)]
        mods += [(s, 2, 1 + (s * j) % 4, 1.0, 1.0, nominal[s] * (0.97 - 0.01 * j), nominal[s] * (1.02 + 0.01 * j))
                 for j in range((s * 5) % 7)]
    return {"n_bins": 64, "bin0": starts, "nominal": nominal, "constrained": [False, True, True, True, False],
            "modifiers": mods, "n_params": 5}


@pytest.mark.parametrize("name", ["odd", "workload"])
def test_last_group_short(name):
    spec = _odd_samples() if name == "odd" else W.binned_model(channels=9, bins=37)
    om, m, alone = B.from_spec(spec), api.BinnedModel(spec), api.BinnedModel(spec)
    rng = np.random.default_rng(6)
    P, most = spec["n_params"], 1023
    if name == "odd":
        th = rng.normal(0.0, 0.3, (most, P))
        th[:, 0] = rng.uniform(0.8, 1.2, most)
    else:
        th = W.binned_toy_thetas(most, 4, P)
    base = om.expected(th[0])[0]
    counts = rng.poisson(np.maximum(base, 0.1), (most, len(base))).astype(float)
    for S in (301, 302, 303, 304, 1023):
        nll, g = m.nll_grad(counts[:S], th[:S])
        for t in (0, 1, 2, 3, 4, S - 4, S - 3, S - 2, S - 1):
            n1, g1 = alone.nll_grad(counts[t], th[t])
            assert n1[0] == nll[t] and np.array_equal(g1[0], g[t]), (S, t)
    for t in (0, 300, 1022):
        ref, rg, scale = om.nll(th[t], counts[t])
        assert abs(nll[t] - ref) <= 1e-12 * scale
        assert np.all(np.abs(g[t] - rg) <= 1e-9 * (np.abs(rg).sum() + np.abs(counts[t]).sum() + 1.0))
