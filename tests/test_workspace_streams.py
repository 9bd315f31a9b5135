"""A dataset's first pass may run on a stream that does not wait for the legacy
stream, on which its buffers are prepared."""
import os

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_preparation_is_waited_for():
    with open(os.path.join(ROOT, "paper_2003_12861_gb300", "csrc", "api.cu")) as fh:
        text = fh.read()
    body = text[text.index("bool ensure_workspace("):text.index("Pass make_pass(")]
    for queued in ("cudaMemset(w.tickets.p", "build_plan(d, all"):
        assert body.index(queued) < body.index("cudaStreamSynchronize(nullptr)")


@pytest.mark.gpu
def test_first_pass_on_a_side_stream_while_the_legacy_stream_is_busy():
    import torch

    from paper_2003_12861_gb300 import api
    from paper_2003_12861_gb300 import workloads as W

    m = api.Model.from_spec(W.decay_model())
    x = np.random.default_rng(1).uniform(0.1, 9.0, 50 * 4096)
    want, want_g = api.nll_grad(m, api.Data.upload(m, [x]), W.DECAY_TRUE)
    side = torch.cuda.Stream()
    th = torch.tensor(W.DECAY_TRUE, device="cuda")
    for _ in range(3):
        d = api.Data.upload(m, [x])
        out = torch.zeros(1, 1 + m.n_free, dtype=torch.float64, device="cuda")
        flags = torch.zeros(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        torch.cuda._sleep(20_000_000)  # about 10 ms on the default (legacy) stream
        api.nll_grad_async(m, d, th, out, flags, stream=side)
        side.synchronize()
        got = out.cpu().numpy()[0]
        assert got[0] == want and np.array_equal(got[1:], want_g)
