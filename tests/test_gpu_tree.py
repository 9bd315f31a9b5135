"""The reduction tree's bits: from a set's per-chunk sums (nll_chunks), the
radix-32 tree of two-sum merges restated in numpy gives exactly the NLL and
gradient of the pass, at chunk counts around the tree's edges (levels that are
left out below 32 children, a second and a third level), with one set, with
several, and with few blocks that take many units each."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _merge(a, b):
    s = a[0] + b[0]
    bb = s - a[0]
    return s, (a[1] + b[1]) + ((a[0] - (s - bb)) + (b[0] - bb))


def _tree(values):
    level = [(v, np.zeros_like(v)) for v in values]
    while len(level) > 1:
        up = []
        for i in range(0, len(level), 32):
            kids = level[i:i + 32] + [(np.zeros_like(values[0]),) * 2] * (32 - len(level[i:i + 32]))
            for o in (16, 8, 4, 2, 1):
                kids = [_merge(kids[k], kids[k ^ o]) for k in range(32)]
            up.append(kids[0])
        level = up
    return level[0][0] + level[0][1]


@pytest.mark.parametrize("blocks_per_sm", [0, 1])
@pytest.mark.parametrize("chunks", [[1], [2], [3], [8], [9], [16], [17], [31], [32], [33], [1025], [5, 1, 33, 2, 17, 70]])
def test_tree_bits(chunks, blocks_per_sm):
    m = api.Model.from_spec(W.gauss_poly1_model())
    m.set_launch(0, blocks_per_sm)
    sizes = [4096 * c - 37 * (k + 1) for k, c in enumerate(chunks)]
    d = api.generate_toys(m, W.GAUSS_POLY1_TRUE, 3, [float(n) for n in sizes], poisson=False)
    for shift in (0.0, 0.01):
        th = W.GAUSS_POLY1_TRUE + shift
        nll, g = api.nll_grad(m, d, th)
        nll, g = np.atleast_1d(nll), np.atleast_2d(g)
        for s, c in enumerate(chunks):
            parts = api.nll_chunks(m, d, th, s)
            assert len(parts) == c
            want = -_tree(list(parts))
            assert nll[s] == want[0] and np.array_equal(g[s], want[1:]), (s, c)
