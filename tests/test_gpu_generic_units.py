"""The generic event kernel at the edges of its work units (parts of a
4096-event chunk; how many depends on the dataset's chunk count) and of the
decay's two branches, against the oracle at the other parity tests'
tolerances; the bits must not depend on the grid, and the pass without
allocations runs the same tree."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

from helpers import check_nll

pytestmark = pytest.mark.gpu

WIDE = np.array([0.9, 0.1, 0.8, -0.2, 0.05, 0.7])  # sigma near tau: z = (sigma/tau - u)/sqrt(2) of both signs
CASES = [("decay_generic_model", W.DECAY_GENERIC_TRUE), ("decay_generic_model", WIDE),
         ("expr_mix_model", W.EXPR_MIX_TRUE)]


@pytest.mark.parametrize("which,th", CASES)
@pytest.mark.parametrize("n", [1, 255, 257, 4096, 57 * 4096 + 1, 113 * 4096 + 300, 229 * 4096 - 1])
def test_units_match_oracle_and_do_not_depend_on_the_grid(oracle_mod, which, th, n):
    import torch

    spec = W.model_for(which)
    om = oracle_mod.Model(spec.nodes, spec.root)
    cols = om.generate(th, 99, 0, 0, n)
    m = api.Model.from_spec(spec)
    d = api.Data.upload(m, cols)
    nll, g = api.nll_grad(m, d, th)
    check_nll(nll, g, om.nll(th, cols), f"{which} n={n}")
    m.set_launch(128, 1)
    nll1, g1 = api.nll_grad(m, d, th)
    assert nll1 == nll and np.array_equal(g1, g)
    m.set_launch(0, 0)
    out = torch.zeros(1 + m.n_free, dtype=torch.float64, device="cuda")
    flags = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.nll_grad_noalloc(m, [torch.from_numpy(c).cuda() for c in cols], torch.tensor(th, device="cuda"), out, flags)
    assert np.array_equal(out.cpu().numpy(), np.concatenate([[nll], g]))


def test_events_outside_the_domain_are_counted_in_every_part():
    spec = W.decay_generic_model()
    m = api.Model.from_spec(spec)
    x = np.full(3 * 4096 + 5, 1.0)
    ok, _ = api.nll_grad(m, api.Data.upload(m, [x]), W.DECAY_GENERIC_TRUE)
    assert np.isfinite(ok)
    for where in (0, 300, 4095, 4096, 3 * 4096 + 4):
        y = x.copy()
        y[where] = np.nan
        nll, _ = api.nll_grad(m, api.Data.upload(m, [y]), W.DECAY_GENERIC_TRUE, allow_domain=True)
        assert nll == np.inf
