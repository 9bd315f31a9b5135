"""hist64's bins on ranges near the smallest floats and with sets around the sizes
at which its kernel changes form, against the FP64 definition."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _model(lo, hi):
    b = W._Builder()
    x = b.obs(lo, hi)
    return api.Model.from_spec(b.spec(b.pdf("poly", x, b.param("a", 0.0, 0.0, 0.0, False))))


def _fractions(x, lo, hi):
    b = np.clip(np.floor((x.astype(np.float64) - lo) * (64.0 / (hi - lo))), 0, 63).astype(np.int64)
    return (np.bincount(b, minlength=64) / float(len(x))).astype(np.float32)


# float's normal numbers end at 1.2e-38
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("lo,hi", [(-1.3e-37, 8.7e-37), (-5.1e-37, 4.9e-37), (-3e-35, 7e-35), (-1e-33, 1e-33), (0.0, 3e-38),
                                   (-2e-39, 1e-38), (-1e-300, 1e-300)])
def test_ranges_near_the_smallest_floats(lo, hi, f32):
    import torch

    m = _model(lo, hi)
    x = np.concatenate([np.linspace(lo, hi, 20001), np.array([0.0, -0.0, 1.1e-38, -1.1e-38, 1e-45, 1.18e-38]),
                        np.linspace(-1.2e-38, 1.2e-38, 4001)])
    x = x[(x >= lo) & (x <= hi)]
    x = x.astype(np.float32) if f32 else x
    out = torch.zeros(1, 64, dtype=torch.float32, device="cuda")
    api.hist64(m, api.Data.upload(m, [x]), 0, out)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy()[0], _fractions(x, lo, hi))


# 511 and 512: the blocks' size; 1023 and 1024: one copy of the counters or 16;
# 2 x 16384 per set on average: one block a set or two
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("sizes", [[511, 0, 63], [512, 1, 0, 65], [1023, 1024, 3], [1], [300] * 700, [40000, 0, 5, 100],
                                   [32767], [32768], [70000, 20000, 8304], [5, 98299]])
def test_set_sizes_around_the_kernels_forms(sizes, f32):
    import torch

    lo, hi = 0.0, 10.0
    m = _model(lo, hi)
    off = np.concatenate([[0], np.cumsum(sizes)])
    x = np.random.default_rng(int(off[-1])).exponential(1.5, off[-1])
    x = x.astype(np.float32) if f32 else x
    out = torch.full((len(sizes), 64), 3.0, dtype=torch.float32, device="cuda")
    api.hist64(m, api.Data.upload(m, [x], offsets=off), 0, out)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    for s in range(len(sizes)):
        part = x[off[s]:off[s + 1]]
        want = _fractions(part, lo, hi) if len(part) else np.zeros(64, dtype=np.float32)
        assert np.array_equal(got[s], want), s
