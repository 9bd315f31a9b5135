"""The generic event kernel on sets that fill only some of their chunks' parts:
every number of parts (it falls with the dataset's chunks), sizes around the
parts' ends, empty sets; against the oracle, and the same bits for every grid
and for the device's own plans of a fit."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

from helpers import check_nll

pytestmark = pytest.mark.gpu

# 22 chunks a copy: 16 parts of 256 events, then 8, 8, 4, 2 and 1
SIZES = [1, 255, 256, 257, 0, 511, 513, 1024, 1025, 1500, 2048, 2049, 4095, 4096, 4097, 6000, 8191, 8193]


@pytest.mark.parametrize("copies", [1, 4, 6, 12, 24, 25])
def test_ragged_sets(oracle_mod, copies):
    spec = W.decay_generic_model()
    om = oracle_mod.Model(spec.nodes, spec.root)
    sizes = SIZES * copies
    off = np.concatenate([[0], np.cumsum(sizes)])
    x = om.generate(W.DECAY_GENERIC_TRUE, 7, 0, 0, int(off[-1]))[0]
    m = api.Model.from_spec(spec)
    d = api.Data.upload(m, [x], offsets=off)
    th = np.array([W.DECAY_GENERIC_TRUE * (1 + 0.001 * (s % 7)) for s in range(len(sizes))])
    nll, g = api.nll_grad(m, d, th)
    for s in list(range(len(SIZES))) + [len(sizes) - 1]:
        if sizes[s] == 0:
            assert nll[s] == 0.0 and np.all(g[s] == 0.0)
        else:
            check_nll(nll[s], g[s], om.nll(th[s], [x[off[s]:off[s + 1]]]), f"set {s} of {sizes[s]}")
    assert np.allclose(api.nll(m, d, th), nll, rtol=1e-13, atol=0.0)
    for blocks in (1, 3):
        m.set_launch(128, blocks)
        a, ga = api.nll_grad(m, d, th)
        assert np.array_equal(a, nll) and np.array_equal(ga, g)
    m.set_launch(0, 0)


def test_fit_rounds_on_the_device_and_the_host_agree():
    m = api.Model.from_spec(W.decay_generic_model())
    off = np.concatenate([[0], np.cumsum([300, 1500, 5000, 900, 4096, 700] * 4)])
    d = api.generate_toys(m, W.DECAY_GENERIC_TRUE, 11, np.diff(off).astype(float), poisson=False)
    a = api.fit(m, d)
    b = api.fit(m, d, device_steps=False)
    for k in ("theta", "nll", "n_evals", "status"):
        assert np.array_equal(a[k], b[k]), k
