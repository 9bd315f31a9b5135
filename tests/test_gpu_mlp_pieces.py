"""The network's products whose K is summed in pieces beside one another in
tensor memory: a number of pieces that is no power of two (400: 3, 2000: 11)
and one that takes all columns (2048: 16), under few output tiles.  Oracle and
tolerances of the other shapes: float64 with the same BF16 rounding, a layer's
gradient to 2e-2 of its largest element and 1e-2 in the 2-norm."""
import numpy as np
import pytest
import torch

from oracle import mlp as M
from paper_2003_12861_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,hidden,layers,n_out,B", [(400, 16, 1, 3, 33), (2000, 24, 1, 5, 20), (2048, 32, 1, 6, 129),
                                                        (12, 2048, 1, 3, 40), (2048, 40, 0, 7, 300)])
def test_gradient_and_forward(n_in, hidden, layers, n_out, B):
    net = api.MLP(n_in, hidden, layers, n_out, seed=5)
    shapes = M.layer_shapes(n_in, hidden, layers, n_out)
    rng = np.random.default_rng(B)
    x = rng.standard_normal((B, n_in)).astype(np.float32)
    t = rng.standard_normal((B, n_out)).astype(np.float32)
    p = net.get_params()
    dx, dt = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    g, again = torch.zeros(net.n_params, device="cuda"), torch.zeros(net.n_params, device="cuda")
    loss = net.grad(dx, dt, g)
    assert net.grad(dx, dt, again) == loss and torch.equal(g, again)
    want_loss, want = M.loss_and_grad(p, x, t, shapes)
    assert abs(loss - want_loss) <= 2e-2 * want_loss
    got, o = g.cpu().numpy().astype(np.float64), 0
    for (i, j) in shapes:
        for n in (i * j, j):
            d, w = got[o:o + n] - want[o:o + n], want[o:o + n]
            assert np.max(np.abs(d)) <= 2e-2 * np.max(np.abs(w)), (i, j, n)
            assert np.linalg.norm(d) <= 1e-2 * np.linalg.norm(w), (i, j, n)
            o += n
    y = torch.zeros(B, n_out, device="cuda")
    net.forward(dx, y)
    ref, _ = M.forward(p, x, shapes)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= 2e-2 * np.max(np.abs(ref))
