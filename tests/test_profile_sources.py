"""The event kernel's source digest covers every file that the kernel is
compiled from: a committed ncu summary does not outlive a change in one."""
import os
import re

import bench

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_12861_gb300", "csrc")


def test_the_digest_covers_what_the_event_kernel_includes():
    seen, todo = set(), ["nll.cu"]
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        with open(os.path.join(CSRC, name)) as fh:
            todo += [f for f in re.findall(r'^#include "([^"/]+)"', fh.read(), re.M)]
    assert seen - {"api_internal.h", "rf.h"} == set(bench.KERNEL_SOURCES)
