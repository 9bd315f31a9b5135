"""A captured pass keeps its buffers when another model's evaluation on the
same dataset grows them."""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_a_datasets_buffers_keep_what_they_had():
    with open(os.path.join(ROOT, "paper_2003_12861_gb300", "csrc", "api_internal.h")) as fh:
        text = fh.read()
    body = text[text.index("struct Workspace {"):]
    kept = re.search(r"GrowBuf ([^;]*);", body).group(1)
    for buf in ("consts", "flags", "tree", "tree_bad", "tickets", "counter", "slow", "ffc", "part_m", "part_fb", "part_info"):
        assert re.search(r"\b%s\b" % buf, kept), buf


@pytest.mark.gpu
@pytest.mark.parametrize("n", [300, 100000])
def test_replay_after_a_larger_model(n):
    import torch

    from paper_2003_12861_gb300 import api
    from paper_2003_12861_gb300 import workloads as W

    b = W._Builder()
    x = b.obs(0.0, 10.0)
    small = api.Model.from_spec(b.spec(b.pdf("exp", x, b.param("c", -0.3, -5.0, 5.0))))
    v = np.random.default_rng(3).uniform(0.1, 9.9, n)
    d = api.Data.upload(small, [v])
    want, want_g = api.nll_grad(small, d, np.array([-0.31]))
    th = torch.tensor([-0.31], dtype=torch.float64, device="cuda")
    out, flags = torch.zeros(1, 2, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        api.nll_grad_async(small, d, th, out, flags, stream=torch.cuda.current_stream())
    large = api.Model.from_spec(W.decay_model())
    for fp64 in (False, True):
        large.set_fp64(fp64)
        a, ga = api.nll_grad(large, d, W.DECAY_TRUE)
        ref, rg = api.nll_grad(large, api.Data.upload(large, [v]), W.DECAY_TRUE)
        assert a == ref and np.array_equal(ga, rg)
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        got = out.cpu().numpy()[0]
        assert got[0] == want and np.array_equal(got[1:], want_g)
    again, _ = api.nll_grad(large, d, W.DECAY_TRUE)
    assert again == a
