"""Kernels are launched while the kernel before them still runs, so what that one
writes is not read-only during their lifetime: no source may load global memory
through the non-coherent path."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_07508_gb300", "csrc")


def test_no_non_coherent_global_loads():
    found = []
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh", ".h")):
            continue
        with open(os.path.join(CSRC, name)) as f:
            code = re.sub(r"//[^\n]*", "", f.read())
        found += [(name, m) for m in re.findall(r"__ldg\b|ld\.global\.nc|const [\w:]+ \*\s*__restrict__", code)]
    assert not found
