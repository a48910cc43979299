"""Kernels launched while the kernel before them still runs (those that call grid_wait) read what that kernel writes: not
through the read-only data path, which is for memory that nothing writes while the kernel is resident."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0910_3915_gb300", "csrc")


def kernels():
    """(name, parameter list, body) of every __global__ function, comments left out."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\(([^{;]*)\)\s*\{", src):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[at], 0)
                at += 1
            yield m.group(1), m.group(2), src[m.end():at]


def test_dependent_kernels_load_plainly():
    dependent = {n: (p, b) for n, p, b in kernels() if re.search(r"\bgrid_wait\(\)", b)}
    assert {"adj_forward_kernel", "adj_local_kernel", "adj_gather_kernel", "angle_kernel", "static_finish_kernel",
            "step_tma_kernel"} <= set(dependent)
    for name, (params, body) in dependent.items():
        assert not re.search(r"const\s+[\w:]+\s*\*\s*__restrict__", params), name
        assert not re.search(r"\b__ldg\(|Codec<S>::load2?\(|const\s+[\w:]+\s*\*\s*__restrict__", body), name
