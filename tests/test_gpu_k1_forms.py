"""The parameter point's two forms (a block or a thread per set) around the
set counts where a pass changes between them: every set's result is that of
the set alone, to the bit."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which,true,edge", [("decay_model", W.DECAY_TRUE, 768), ("gauss_poly1_model", W.GAUSS_POLY1_TRUE, 384),
                                             ("prod3_model", W.PROD3_TRUE, 768), ("decay_generic_model", W.DECAY_GENERIC_TRUE, 768)])
def test_forms_agree_bit_for_bit(which, true, edge):
    m = api.Model.from_spec(W.model_for(which))
    th = W.toy_thetas(edge + 1, 11, true, 0.03)
    # every dataset holds the same number of chunks in all, so that the event
    # units are the same: sets beyond `edge` are empty in the smaller one
    mean = np.full(edge + 1, 40.0)
    many = api.generate_toys(m, true, 5, mean, poisson=False)
    cols = [many.read(c, 0, many.offsets()[-1]) for c in range(W.model_for(which).n_obs)]
    fewer = api.Data.upload(m, cols, offsets=many.offsets()[:-2].tolist() + [int(many.offsets()[-1])])
    a, ga = api.nll_grad(m, many, th)
    b, gb = api.nll_grad(m, fewer, th[:-1])
    assert np.array_equal(a[:edge - 1], b[:edge - 1]) and np.array_equal(ga[:edge - 1], gb[:edge - 1])
    assert np.all(np.isfinite(a)) and np.all(np.isfinite(b))
