"""hist64's float bins against the FP64 definition: bitwise the same counts for
values on and beside the bin edges, outside the range, not finite and random,
in FP64 and FP32 columns, with one block a set and with several."""
import numpy as np
import pytest

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _values(lo, hi, n, f32):
    rng = np.random.default_rng(int(n) + 1)
    edges = lo + (hi - lo) * np.arange(65) / 64
    near = np.concatenate([edges, np.nextafter(edges, -np.inf), np.nextafter(edges, np.inf),
                           edges * (1 + 3e-7), edges * (1 - 3e-7)])
    odd = np.array([np.nan, np.inf, -np.inf, 0.0, -0.0, 1e300, -1e300, 1e-300, lo - 1e9, hi + 1e9, 5e-324, 3e38,
                    lo - 64 * (hi - lo), hi + 2 * (hi - lo)])
    x = np.concatenate([odd, near, rng.uniform(lo - 0.1, hi + 0.1, n)])
    with np.errstate(over="ignore"):
        return x.astype(np.float32) if f32 else x


def _counts(x, lo, hi):
    t = np.floor((x.astype(np.float64) - lo) * (64.0 / (hi - lo)))
    # as the device converts: NaN to 0, out of range saturated
    b = np.clip(np.nan_to_num(t, nan=0.0, posinf=63, neginf=0), 0, 63).astype(np.int64)
    return np.bincount(b, minlength=64)


# 16384 events per block of a set: one block below 32768, then several
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("n", [1, 2047, 32000, 33000, 400001])
@pytest.mark.parametrize("lo,hi", [(0.0, 10.0), (5.2, 5.4), (-1.0, 1.0), (5000.0, 5000.5)])
def test_bins(lo, hi, n, f32):
    import torch

    b = W._Builder()
    x = b.obs(lo, hi)
    spec = b.spec(b.pdf("poly", x, b.param("a", 0.0, 0.0, 0.0, False)))
    m = api.Model.from_spec(spec)
    v = _values(lo, hi, n, f32)
    d = api.Data.upload(m, [v], offsets=[0, 0, len(v)])
    out = torch.full((2, 64), 7.0, dtype=torch.float32, device="cuda")
    api.hist64(m, d, 0, out)
    torch.cuda.synchronize()
    h = out.cpu().numpy()
    assert np.array_equal(h[0], np.zeros(64, dtype=np.float32))
    want = (_counts(v, lo, hi) / float(len(v))).astype(np.float32)
    assert np.array_equal(h[1], want)
