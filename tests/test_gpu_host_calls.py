"""Host-buffer calls on both sides of the sizes up to which their results
come without copies of their own, bit for bit what the device-resident calls
give, with an empty set, a set outside the domain and (in turn) calls of
different sizes on one dataset's buffers."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sets", [1, 2, 1170, 1171])  # 7 doubles a set: 64 KiB lies between the last two
@pytest.mark.parametrize("which,true", [("decay_model", W.DECAY_TRUE), ("decay_generic_model", W.DECAY_GENERIC_TRUE)])
def test_likelihood_call(which, true, sets):
    import torch

    m = api.Model.from_spec(W.model_for(which))
    rng = np.random.default_rng(4)
    sizes = np.arange(sets) * 7 % 300 + 5
    if sets > 1:
        sizes[1] = 0
    off = np.concatenate([[0], np.cumsum(sizes)])
    d = api.Data.upload(m, [rng.uniform(0.1, 9.0, off[-1])], offsets=off)
    for step in (0.0, 0.01):
        th = np.tile(np.asarray(true) * (1 + step), (sets, 1))
        if sets > 2:
            th[2, 0] = -1.0  # tau < 0
        out = torch.zeros(sets, 1 + m.n_free, dtype=torch.float64, device="cuda")
        flags = torch.zeros(sets, dtype=torch.int32, device="cuda")
        api.nll_grad_async(m, d, torch.tensor(th, device="cuda"), out, flags)
        ref = out.cpu().numpy()
        nll, g = api.nll_grad(m, d, th, allow_domain=True)
        nll, g = np.atleast_1d(nll), np.atleast_2d(g)
        only = np.atleast_1d(api.nll(m, d, th, allow_domain=True)) if sets == 1 else nll
        good = np.arange(sets) != 2
        assert np.array_equal(nll[good], ref[good, 0]) and np.array_equal(g[good], ref[good, 1:])
        assert np.allclose(only[good], nll[good], rtol=1e-12)
        assert sets <= 2 or (nll[2] == np.inf and int(flags[2]) != 0)
        assert sets == 1 or nll[1] == 0.0


def test_binned_call():
    import torch

    m = api.BinnedModel(W.binned_model(channels=9, bins=37))
    limit = (256 << 10) // 8  # doubles of counts, parameters and results in one buffer
    n = limit // (m.n_bins + 2 * m.n_params + 1)
    for sets in (1, n, n + 1, 2):
        rng = np.random.default_rng(sets)
        counts = rng.poisson(50.0, (sets, m.n_bins)).astype(np.float64)
        th = np.tile(np.where(np.arange(m.n_params) < 3, 1.0, 0.0), (sets, 1)) + rng.uniform(-0.01, 0.01, (sets, m.n_params))
        out = torch.zeros(sets, 1 + m.n_params, dtype=torch.float64, device="cuda")
        flags = torch.zeros(sets, dtype=torch.int32, device="cuda")
        m.nll_grad_async(torch.tensor(counts, device="cuda"), torch.tensor(th, device="cuda"), out, flags)
        ref = out.cpu().numpy()
        nll, g = m.nll_grad(counts, th)
        assert np.array_equal(np.atleast_1d(nll), ref[:, 0]) and np.array_equal(np.atleast_2d(g), ref[:, 1:])
