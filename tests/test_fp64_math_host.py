"""The error of the generic event kernel's exponential and error functions
(csrc/fp64_math.cuh) in units in the last place, compiled for the host and
compared with mpmath over their tables, at the tables' points, beside the
points where the nearest one changes, and at random.

Bounds: the result is one addition of a table value and a small term, so half
a unit plus the term's own error, doubled for a result just below a power of
two.  exp's term is at most h = ln2/512 of the value, its roundings below 0.01,
and its polynomial leaves h^5/480 (r^5/120 economised by a Chebyshev polynomial
of degree 3, 1/4): 0.5 + 0.085 + 0.01.  erfc's and erfcx's terms are at most
1/16 of a logarithmic derivative of up to 1.13 (0.5 + 2 * 0.07 * 1.2 < 0.7)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2003_12861_gb300", "csrc")


def _run(tmp_path, lines):
    gxx, cuda = shutil.which("g++"), os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if gxx is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no g++ or no CUDA headers")
    exe = str(tmp_path / "fp64_math_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC, "-I", os.path.join(cuda, "include"),
                    os.path.join(ROOT, "tests", "native", "fp64_math_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], input="".join(lines), check=True, capture_output=True, text=True).stdout
    return [float.fromhex(v) for v in out.split()]


def _beside(points):
    p = np.asarray(points)
    return np.concatenate([p, np.nextafter(p, -np.inf), np.nextafter(p, np.inf)])


@pytest.mark.parametrize("which", ["e", "l", "r"])
def test_error_in_units_in_the_last_place(tmp_path, which):
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 160
    rng = np.random.default_rng(12)
    if which == "e":
        step = np.log(2.0) / 256
        x = np.concatenate([_beside(step * np.arange(-300, 301)), _beside(step * (np.arange(-300, 300) + 0.5)),
                            rng.uniform(-700.0, 700.0, 1500), rng.uniform(-1.0, 1.0, 1500), 10.0 ** rng.uniform(-20, 0, 200),
                            [0.0, -0.0, 707.9, -707.9]])
        exact, bound = mp.exp, 0.5 + (np.log(2.0) / 512) ** 5 / 480 / 2.0**-53 + 0.01
    elif which == "l":
        x = np.concatenate([_beside(-np.arange(0, 56) / 8.0), _beside(-(np.arange(0, 56) + 0.5) / 8.0),
                            rng.uniform(-7.0, 0.0, 2000), -(10.0 ** rng.uniform(-20, 0, 200))])
        x = x[(x <= 0.0) & (x > -7.0)]
        exact, bound = mp.erfc, 0.7
    else:
        x = np.concatenate([_beside(np.arange(1, 64) / 8.0), _beside((np.arange(0, 63) + 0.5) / 8.0),
                            rng.uniform(0.0, 8.0, 2000), 10.0 ** rng.uniform(-20, 0, 200)])
        x = x[(x > 0.0) & (x < 8.0)]
        exact, bound = (lambda v: mp.exp(v * v) * mp.erfc(v)), 0.7
    got = _run(tmp_path, [f"{which} {v.hex()}\n" for v in x.tolist()])
    assert len(got) == len(x)
    worst = max(float(abs(mp.mpf(g) - exact(mp.mpf(v)))) / np.spacing(float(exact(mp.mpf(v)))) for v, g in zip(x.tolist(), got))
    assert worst <= bound, worst


def test_ends_of_the_tables(tmp_path):
    lines = ["l -7.07\n", "l -7.5\n", "l -30\n", "e 710\n", "e -746\n", "e inf\n", "e -inf\n", "e nan\n"]
    got = _run(tmp_path, lines)
    assert got[:3] == [2.0, 2.0, 2.0] and got[3] == np.inf and got[4] == 0.0 and got[5] == np.inf and got[6] == 0.0
    assert np.isnan(got[7])
