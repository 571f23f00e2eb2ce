"""Every kernel of the library may be launched while its predecessor in the
stream still runs (programmatic dependent launch), so each must begin by
waiting for it: the first statement of every __global__ function is pdl_wait().
Read from the sources; no GPU needed."""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1803_00417_gb300", "csrc")


def _close(s, i):
    depth = 0
    for k in range(i, len(s)):
        depth += (s[k] == "(") - (s[k] == ")")
        if depth == 0:
            return k + 1
    raise AssertionError("unbalanced parentheses")


def _kernels(path):
    with open(path) as f:
        s = re.sub(r"//[^\n]*", "", f.read())
    for m in re.finditer(r"__global__", s):
        i = m.end()
        while True:  # past __launch_bounds__(...) and the like to the kernel's own parameters
            j = s.index("(", i)
            name = re.search(r"(\w+)\s*$", s[i:j]).group(1)
            i = _close(s, j)
            if not name.startswith("__"):
                break
        if s[i:].lstrip().startswith("{"):
            yield name, s[s.index("{", i) + 1:].lstrip()


def test_every_kernel_waits_first():
    names = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for name, body in _kernels(path):
            names.append(name)
            assert re.match(r"(hb::)?pdl_wait\(\);", body), (os.path.basename(path), name)
    assert len(names) > 90, len(names)
