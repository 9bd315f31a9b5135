"""The generic kernel's own exponential and error functions where they change
branch (arguments beyond their tables, steps at the table's points), against
the oracle at the other parity tests' tolerances."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W
from paper_2003_12861_gb300.workloads import Node

from helpers import check_nll

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau,mu,sigma", [(0.06, 0.1, 1.0), (0.25, -0.4, 0.9), (1.0, 0.5, 0.05), (9.0, 0.0, 0.3)])
def test_decay_over_the_tables_ends(oracle_mod, tau, mu, sigma):
    spec = W.decay_generic_model()
    om = oracle_mod.Model(spec.nodes, spec.root)
    th = np.array([tau, mu, sigma, -0.2, 0.05, 0.5])
    # z = (sigma/tau - (t - mu)/sigma) / sqrt 2 at the points of the table, halfway between them, and beyond
    z = np.concatenate([np.arange(-120, 160) / 16.0, np.linspace(-9.0, 14.0, 997)])
    t = mu + sigma * (sigma / tau - np.sqrt(2.0) * z)
    t = t[(t > 0.0) & (t < 10.0)]
    m = api.Model.from_spec(spec)
    nll, g = api.nll_grad(m, api.Data.upload(m, [t]), th)
    check_nll(nll, g, om.nll(th, [t]), f"tau {tau} sigma {sigma}")


@pytest.mark.parametrize("sigma,c", [(0.01, -0.6), (0.3, -150.0), (2.0, 140.0)])
def test_exponentials_beyond_the_table(oracle_mod, sigma, c):
    nodes = [Node("obs", (), 0, -1.0, 4.0), Node("param", (), -0.6, -200, 200, True),
             Node("param", (), 1.0, -5, 5, True), Node("param", (), 0.3, 0.001, 5, True),
             Node("exp", (0, 1)), Node("gauss", (0, 2, 3)), Node("param", (), 0.5, 0, 1, True),
             Node("sum", (4, 5, 6))]
    om = oracle_mod.Model(nodes, 7)
    th = np.array([c, 1.0, sigma, 0.5])
    x = np.linspace(-0.999, 3.999, 5003)
    if sigma < 0.1:  # the Gaussian underflows far from its mean; the exponential carries the sum
        assert np.exp(-0.5 * ((x[0] - 1.0) / sigma) ** 2) == 0.0
    m = api.Model(nodes, 7)
    nll, g = api.nll_grad(m, api.Data.upload(m, [x]), th)
    ref = om.nll(th, [x])
    if c > 100:  # the oracle's d/dc overflows there: its values of the mirrored problem, x -> 3 - x
        mirrored = om.nll(np.array([-c, 2.0, sigma, 0.5]), [3.0 - x])
        assert abs(mirrored[0] - ref[0]) <= 1e-12 * ref[2]
        sign = np.array([-1.0, -1.0, 1.0, 1.0])
        ref = (mirrored[0], sign * mirrored[1], mirrored[2], mirrored[3], mirrored[4])
    check_nll(nll, g, ref, f"sigma {sigma} c {c}")
