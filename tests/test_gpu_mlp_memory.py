"""A network call that finds no memory fails and leaves the network usable."""
import ctypes as C

import pytest
import torch

from paper_2003_12861_gb300 import _lib as L
from paper_2003_12861_gb300 import api

pytestmark = pytest.mark.gpu


def test_smaller_batches_after_one_without_memory():
    net = api.MLP(seed=3)
    x, t = torch.rand(300, 64, device="cuda"), torch.randn(300, 6, device="cuda")
    y, again = torch.zeros(300, 6, device="cuda"), torch.zeros(300, 6, device="cuda")
    g, g2 = torch.zeros(net.n_params, device="cuda"), torch.zeros(net.n_params, device="cuda")
    net.forward(x, y)
    loss = net.grad(x, t, g)
    lib = L.load()
    for _ in range(2):  # 1.6e12 bytes of activations: refused before anything is read or launched
        s = lib.rf_mlp_forward(net._h, C.c_void_p(x.data_ptr()), 1 << 30, C.c_void_p(y.data_ptr()), None)
        assert s == L.RF_E_OOM
        net.forward(x, again)
        assert net.grad(x, t, g2) == loss
        torch.cuda.synchronize()
        assert torch.equal(y, again) and torch.equal(g, g2)
