"""The generator's float filter and event pools against the oracle, which takes
every accept/reject decision in FP64: bitwise the same events for every form
that a filter term has (each leaf kind, more than two Chebychev terms, nested
sums, fractions of exactly 0 and 1, narrow peaks far from zero, wide ranges)
and for the forms without one (Poisson and program leaves), at sizes around
the pools' edges and over many small sets."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _model(lo, hi, make):
    b = W._Builder()
    x = b.obs(lo, hi)
    p = lambda v: b.param("p", v, 0.0, 0.0, False)  # noqa: E731
    return b.spec(make(b, x, p))


FORMS = {
    "gauss": (-3.0, 4.0, lambda b, x, p: b.pdf("gauss", x, p(0.3), p(0.8))),
    "narrow_peak": (5278.0, 5281.0, lambda b, x, p: b.pdf(
        "sum", b.pdf("gauss", x, p(5279.3), p(1e-4)), b.pdf("poly", x, p(0.0)), p(0.6))),
    "exp_up": (0.0, 40.0, lambda b, x, p: b.pdf("exp", x, p(0.7))),
    "exp_down": (-20.0, 5.0, lambda b, x, p: b.pdf("exp", x, p(-1.3))),
    "decay_wide_resolution": (-6.0, 9.0, lambda b, x, p: b.pdf("gaussexp", x, p(0.4), p(-0.5), p(1.7))),
    "decay_narrow_resolution": (-0.01, 10.0, lambda b, x, p: b.pdf("gaussexp", x, p(1.5), p(0.002), p(0.004))),
    "decay_long_resolution": (-40.0, 3.0, lambda b, x, p: b.pdf("gaussexp", x, p(0.05), p(2.0), p(6.0))),
    "cheb7": (-2.0, 5.0, lambda b, x, p: b.pdf("cheb", x, *[p(v) for v in (0.3, -0.2, 0.1, 0.05, -0.1, 0.02, 0.04)])),
    "cheb1": (5.2, 5.4, lambda b, x, p: b.pdf("cheb", x, p(-0.9))),
    "poly7": (-1.5, 2.0, lambda b, x, p: b.pdf("poly", x, *[p(v) for v in (0.1, 0.5, 0.02, 0.1, 0.0, 0.01, 0.001)])),
    "flat": (0.0, 7.0, lambda b, x, p: b.pdf("poly", x, p(0.0))),
    "nested": (0.0, 10.0, lambda b, x, p: b.pdf(
        "sum", b.pdf("sum", b.pdf("gauss", x, p(2.0), p(0.3)), b.pdf("gauss", x, p(7.0), p(0.1)), b.pdf("exp", x, p(-0.4)),
                     p(0.2), p(0.5)), b.pdf("cheb", x, p(0.1), p(0.2), p(-0.1)), p(0.7))),
    "fraction_0": (0.0, 10.0, lambda b, x, p: b.pdf("sum", b.pdf("gauss", x, p(3.0), p(0.2)), b.pdf("exp", x, p(-0.3)), p(0.0))),
    "fraction_1": (0.0, 10.0, lambda b, x, p: b.pdf("sum", b.pdf("gauss", x, p(3.0), p(0.2)), b.pdf("exp", x, p(-0.3)), p(1.0))),
    "poisson": (0.0, 20.0, lambda b, x, p: b.pdf("poisson", x, p(4.5))),
    "program": (0.2, 5.0, lambda b, x, p: b.expr("x p0 pow x p1 * neg exp *", (), x, p(1.5), p(1.2))),
}


@pytest.mark.parametrize("form", sorted(FORMS))
def test_every_form_matches_the_oracle(oracle_mod, form):
    spec = _model(*FORMS[form])
    m = api.Model.from_spec(spec)
    om = oracle_mod.Model(spec.nodes, spec.root)
    n = 5003
    d = api.generate_toys(m, None, 0xABCD_0123_4567, [float(n), 700.0], poisson=False)
    got = d.read(0)
    th = np.zeros(0)
    assert np.array_equal(got[:n], om.generate(th, 0xABCD_0123_4567, 0, 0, n)[0])
    assert np.array_equal(got[n:], om.generate(th, 0xABCD_0123_4567, 1, 0, 700)[0])


# 32 events a pool up to 32 x 32 x 152 events, 64 beyond: around the first
# step, and odd ends of a pool.
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 155647, 155649, 311297])
def test_pool_edges(oracle_mod, n):
    spec = W.gauss_poly1_model()
    m = api.Model.from_spec(spec)
    om = oracle_mod.Model(spec.nodes, spec.root)
    th = W.GAUSS_POLY1_TRUE
    got = api.generate_toys(m, th, 5, [float(n)], poisson=False).read(0)
    i0 = max(0, n - 2000)
    assert np.array_equal(got[i0:], om.generate(th, 5, 0, i0, n)[0])
    assert np.array_equal(got[:min(n, 2000)], om.generate(th, 5, 0, 0, min(n, 2000))[0])


def test_many_small_sets(oracle_mod):
    # pools that span many sets, empty ones among them
    spec = W.prod3_model()
    m = api.Model.from_spec(spec)
    om = oracle_mod.Model(spec.nodes, spec.root)
    sizes = np.random.default_rng(3).integers(0, 9, 400)
    sizes[[0, 7, 8, 399]] = 0
    d = api.generate_toys(m, W.PROD3_TRUE, 77, sizes.astype(float), poisson=False)
    off = d.offsets()
    assert np.array_equal(np.diff(off), sizes)
    cols = [d.read(c) for c in range(3)]
    for s in range(400):
        if sizes[s]:
            want = om.generate(W.PROD3_TRUE, 77, s, 0, int(sizes[s]))
            for c in range(3):
                assert np.array_equal(cols[c][off[s]:off[s + 1]], want[c]), (s, c)
