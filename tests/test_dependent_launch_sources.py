"""Kernels launched with launch_after run beside the kernel before them: only
the call's input (the parameter P, which no kernel of the call writes) may be
__restrict__, because restricted pointers may be read with read-only loads."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1508_05931_gb300", "csrc")


def test_restrict_only_on_the_input():
    text = "\n".join(open(p).read() for p in sorted(glob.glob(os.path.join(CSRC, "*.cu"))))
    kernels = set(re.findall(r"launch_after\(\s*(\w+)", text))
    assert {"k1_poly", "k_cand", "k_star"} <= kernels
    for k in kernels:
        m = re.search(r"__global__[^;{]*?\b%s\(([^)]*)\)" % k, text)
        assert m, k
        named = re.findall(r"__restrict__\s+(\w+)", m.group(1))
        assert set(named) <= {"P"}, (k, named)
