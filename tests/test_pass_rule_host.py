"""Which passes of a fit run beside another one, and so take the parameter
point's form measured for that: the two halves of a pipelined fit alone
(fit.cpp's groups 0 and 1), not its whole-batch passes and device rounds."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2003_12861_gb300", "csrc")


def test_only_a_fits_halves_run_beside_another_pass(tmp_path):
    with open(os.path.join(CSRC, "api.cu")) as fh:
        assert "pass.beside = slot_beside(slot)" in fh.read()
    gxx, cuda = shutil.which("g++"), os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if gxx is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no g++ or no CUDA headers")
    exe = str(tmp_path / "pass_rule_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-I",
                    os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "native", "pass_rule_check.cpp"),
                    "-c", "-o", exe + ".o"], check=True)
    subprocess.run([gxx, exe + ".o", "-o", exe, "-Wl,--unresolved-symbols=ignore-all"], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    assert [tuple(map(int, line.split())) for line in out.splitlines()] == [(-1, 0), (0, 1), (1, 1), (2, 0), (3, 0)]
