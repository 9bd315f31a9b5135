"""The sizes of a dataset's evaluation buffers (csrc/workspace.h), checked on
the CPU against what the event kernels index when models of different sizes
are evaluated on one dataset in turn; and that a call asks for every one of
them, whatever model came before."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2003_12861_gb300", "csrc")


def test_every_part_record_has_room(tmp_path):
    gxx, cuda = shutil.which("g++"), os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if gxx is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no g++ or no CUDA headers")
    exe = str(tmp_path / "workspace_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-I",
                    os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "native", "workspace_check.cpp"),
                    "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    lost = dict(tuple(map(int, line.split())) for line in out.splitlines())
    assert len(lost) == 15 and all(v == 0 for v in lost.values()), lost


def test_a_call_asks_for_every_buffer_of_its_model():
    with open(os.path.join(CSRC, "api.cu")) as fh:
        text = fh.read()
    body = text[text.index("bool ensure_workspace("):text.index("Pass make_pass(")]
    asked = body.index("w.part_info.ensure(")
    assert "return true" not in body[:asked]  # no early way out before the sizes are compared
    for buf in ("consts", "theta", "out", "flags", "tree", "tree_bad", "ffc", "part_m", "part_fb", "part_info", "h_theta",
                "h_out", "h_flags", "tickets"):
        assert re.search(r"w\.%s\.ensure\(" % buf, body), buf
