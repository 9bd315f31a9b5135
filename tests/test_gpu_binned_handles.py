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


def test_memory_grows_with_the_datasets_of_a_call():
    spec = W.binned_model()
    api.BinnedModel(spec)  # the kernels are loaded
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    held = [api.BinnedModel(spec) for _ in range(4)]
    # the coefficients in their three layouts (11 MB) and a few datasets' intermediate results (8 MB)
    assert (free - torch.cuda.mem_get_info()[0]) / 4 < 40e6
    one, th = _points(held[0], spec, 1, 3)
    many, many_th = _points(held[0], spec, 1100, 4)
    first = held[0].nll_grad(one, th)
    whole = held[0].nll_grad(many, many_th)
    for t in (0, 49, 50, 51, 1023, 1024, 1099):
        n, g = held[1].nll_grad(many[t], many_th[t])
        assert n[0] == whole[0][t] and np.array_equal(g[0], whole[1][t])
    nu = [torch.zeros(1100, held[0].n_bins, dtype=torch.float64, device="cuda") for _ in range(2)]
    held[0].expected(torch.tensor(many_th, device="cuda"), nu[0])
    for t in range(3):  # one dataset, then a few, then all
        held[1].expected(torch.tensor(many_th[:(1, 5, 1100)[t]], device="cuda"), nu[1])
    torch.cuda.synchronize()
    assert torch.equal(nu[0], nu[1]) and float(nu[0].min()) > 0.0
    again = held[0].nll_grad(one, th)
    assert np.array_equal(first[0], again[0]) and np.array_equal(first[1], again[1])


def test_a_captured_pass_outlives_the_growth():
    spec = W.binned_model(channels=9, bins=37)
    m = api.BinnedModel(spec)
    counts, th = _points(m, spec, 700, 5)
    want = m.nll_grad(counts, th)
    fresh = api.BinnedModel(spec)  # its first pass is a captured one, of more datasets than it has room for
    c, t = torch.tensor(counts, device="cuda"), torch.tensor(th, device="cuda")
    out = torch.zeros(700, 1 + m.n_params, dtype=torch.float64, device="cuda")
    flags = torch.zeros(700, dtype=torch.int32, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        fresh.nll_grad_async(c, t, out, flags, stream=torch.cuda.current_stream())
    more, more_th = _points(m, spec, 1500, 6)
    grown = fresh.nll_grad(more, more_th)
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        assert np.array_equal(got[:, 0], want[0]) and np.array_equal(got[:, 1:], want[1])
    ref = m.nll_grad(more, more_th)
    assert np.array_equal(ref[0], grown[0]) and np.array_equal(ref[1], grown[1])


def test_more_datasets_than_a_pass_takes():
    spec = _one_bin()
    m, one = api.BinnedModel(spec), api.BinnedModel(spec)
    counts, th = _points(m, spec, 2 * 32768 + 5, 8)
    nll, g = m.nll_grad(counts, th)
    for t in (0, 1, 32767, 32768, 65535, 65536, 65540):
        n, h = one.nll_grad(counts[t], th[t])
        assert n[0] == nll[t] and np.array_equal(h[0], g[t]), t
    back, gb = one.nll_grad(counts[::-1], th[::-1])
    assert np.array_equal(back[::-1], nll) and np.array_equal(gb[::-1], g)
