"""The network's grouped launches at the sizes where they can go wrong: widths
that are no multiple of 4, 8, 16 or 32 and rows that are no multiple of 128
(edge tiles and rows without 16-byte loads), inputs off a 16-byte boundary,
K in several pieces beside one another in tensor memory (a wide layer under
few rows) and over blocks (batches beyond 128 rows, with pieces above 128 at
2100), no hidden layer, and y written over x.  Against the float64 oracle with
the same BF16 rounding; an activation on the other side of a rounding boundary
moves its sample by one BF16 ulp (2^-8), so a layer's gradient may be off by
2e-2 of its largest element and 1e-2 in the 2-norm."""
import numpy as np
import pytest
import torch

from oracle import mlp as M
from paper_2003_12861_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,hidden,layers,n_out,B,skip", [
    (64, 128, 3, 6, 1, 0), (64, 128, 3, 6, 127, 1), (64, 128, 3, 6, 129, 0), (64, 128, 3, 6, 2100, 0),
    (5, 33, 2, 3, 70, 0), (7, 1, 1, 1, 300, 0), (64, 96, 4, 6, 513, 3), (64, 256, 2, 6, 300, 0),
    (40, 300, 2, 10, 260, 0), (64, 16, 0, 6, 400, 0), (300, 16, 1, 40, 33, 0),
])
def test_gradient_and_forward(n_in, hidden, layers, n_out, B, skip):
    net = api.MLP(n_in, hidden, layers, n_out, seed=4)
    shapes = M.layer_shapes(n_in, hidden, layers, n_out)
    rng = np.random.default_rng(B)
    p = net.get_params() + (0.05 * rng.standard_normal(net.n_params)).astype(np.float32)
    net.set_params(p)
    x = rng.standard_normal((B, n_in)).astype(np.float32)
    t = rng.standard_normal((B, n_out)).astype(np.float32)
    dx = torch.zeros(B * n_in + skip, device="cuda")[skip:].view(B, n_in)
    dx.copy_(torch.from_numpy(x))
    dt = torch.from_numpy(t).cuda()
    g = torch.zeros(net.n_params, device="cuda")
    loss = net.grad(dx, dt, g)
    again = torch.zeros_like(g)
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


def test_one_layer_over_its_input():
    net = api.MLP(32, 8, 0, 32, seed=2)
    x = torch.randn(700, 32, device="cuda")
    y = torch.zeros_like(x)
    net.forward(x, y)
    net.forward(x, x)
    torch.cuda.synchronize()
    assert torch.equal(x, y)
