"""A committed DRAM-traffic figure is valid for the sources that the encoder kernels are
built from: the bench's list of them holds every file they include (CPU only)."""
import os
import re

import bench

CSRC = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_2308_05199_gb300", "csrc")


def test_list_is_complete():
    todo, seen = ["zc_kenc.cu", "zc_kbatch.cu"], set()
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        with open(os.path.join(CSRC, name)) as f:
            todo += [i for i in re.findall(r'#include "(\w+\.\w+)"', f.read())
                     if os.path.exists(os.path.join(CSRC, i))]
    assert seen == set(bench.ENCODER_SOURCES)
