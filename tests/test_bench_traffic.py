"""The DRAM traffic that bench.py scales to the step's stencil launches was captured from the kernel of those launches, and
its hash covers every header of the kernel."""
import json
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_1701_00726_gb300", "csrc")


def test_capture_is_of_the_solvers_stencil():
    d = json.load(open(os.path.join(bench.ROOT, "profiles", "bri_stencil_traffic.txt")))
    assert all(k.startswith(bench.STENCIL_KERNEL + "<") for k in d["kernels"])
    text = {f: open(os.path.join(CSRC, f)).read() for f in bench.STENCIL_SOURCES}
    home = [f for f, t in text.items() if re.search(rf"^ +{bench.STENCIL_KERNEL}\(", t, re.M)]
    assert home == ["packed_solve.cuh"]
    for t in text.values():  # headers that hold device code of it (internal.cuh: host declarations)
        for inc in re.findall(r'#include "([a-z0-9_]+\.cuh)"', t):
            assert inc in bench.STENCIL_SOURCES or inc == "internal.cuh", inc
    apply = open(os.path.join(CSRC, "mscg.cu")).read()
    assert bench.STENCIL_KERNEL + "<" in apply  # launched by the solver
