"""One dataset evaluated with models of different sizes in turn (its buffers
are shared): every result is bit for bit that of a dataset of its own, with
the interpreter's part records, the float-float ones and their fallback
events, NLL alone and with the gradient."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _exponential():
    b = W._Builder()
    x = b.obs(0.0, 10.0)
    return b.spec(b.pdf("exp", x, b.param("c", -0.3, -5.0, 5.0)))


def _models():
    """name -> (model, theta), all on one observable in [0, 10]."""
    out = {"exp": (api.Model.from_spec(_exponential()), np.array([-0.31]))}
    for name, spec, th in (("decay", W.decay_model, W.DECAY_TRUE), ("line", W.gauss_poly1_model, W.GAUSS_POLY1_TRUE)):
        for fp64 in (False, True):
            m = api.Model.from_spec(spec())
            if fp64:
                m.set_fp64(True)
            out[name + ("_fp64" if fp64 else "")] = (m, th * 1.01)
    return out


ORDERS = [("exp", "decay", "decay_fp64", "decay"), ("line", "decay_fp64", "decay", "exp"),
          ("line_fp64", "decay", "decay_fp64", "line"), ("decay_fp64", "exp", "decay_fp64", "line_fp64")]


@pytest.mark.parametrize("order", ORDERS)
@pytest.mark.parametrize("n", [5, 4097, 66 * 4096 + 9, 250000])
def test_models_in_turn_on_one_dataset(order, n):
    rng = np.random.default_rng(n)
    x = rng.uniform(0.0, 10.0, n)
    x[: n // 2] = rng.exponential(1.5, n // 2) % 10.0
    models = _models()
    shared = api.Data.upload(models["exp"][0], [x])
    for name in order + order:
        m, th = models[name]
        own = api.Data.upload(m, [x])
        a, ga = api.nll_grad(m, shared, th)
        b, gb = api.nll_grad(m, own, th)
        assert a == b and np.array_equal(ga, gb), name
        assert api.nll(m, shared, th) == api.nll(m, own, th), name


def test_set_fp64_switched_on_one_model():
    x = np.random.default_rng(2).uniform(0.0, 10.0, 70000)
    first = api.Model.from_spec(_exponential())
    d = api.Data.upload(first, [x], offsets=[0, 30000, 30000, 70000])
    m = api.Model.from_spec(W.decay_model())
    th = np.tile(W.DECAY_TRUE, (3, 1))
    api.nll_grad(first, d, np.full((3, 1), -0.2))
    api.nll_grad(m, d, th)
    for fp64 in (True, False, True):
        m.set_fp64(fp64)
        a, ga = api.nll_grad(m, d, th)
        b, gb = api.nll_grad(m, api.Data.upload(m, [x], offsets=[0, 30000, 30000, 70000]), th)
        assert np.array_equal(a, b) and np.array_equal(ga, gb)
