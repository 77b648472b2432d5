"""Loads of the stage kernels that start before the stage they depend on ends.

A kernel launched as a programmatic dependent runs while the stage that writes
its input is still running, so that input is not read-only for the kernel's
lifetime: the non-coherent load path and `__restrict__` views of it, which
allow the loads to move above the wait, are excluded there.  Host only: the
kernel sources are read."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1607_03399_gb300", "csrc")


def _kernels():
    """{name: body} of every __global__ function of the stage sources."""
    out = {}
    for name in ("kernels.cuh", "stage_split.cuh", "adjoint_kernels.cuh"):
        with open(os.path.join(CSRC, name)) as f:
            src = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", src):
            i = src.index("{", m.end())
            depth, j = 1, i + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[j], 0)
                j += 1
            out[m.group(1)] = src[i:j]
    return out


def test_dependent_stages_read_their_input_with_ordinary_loads():
    kernels = _kernels()
    dependents = {k for k, b in kernels.items() if "pdl_wait()" in b}
    assert {"k_wedge_stage", "k_wedge_wide"} <= dependents
    for k in dependents:
        for word in ("ldg4(", "__ldg(", "__restrict__", "ld.global.nc"):
            assert word not in kernels[k], (k, word)


def test_only_kernels_that_wait_are_launched_as_dependents():
    kernels = _kernels()
    with open(os.path.join(CSRC, "kernels.cuh")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    assert src.count("cudaLaunchAttributeProgrammaticStreamSerialization") == 1
    launches = re.findall(r"launch_dependent\((\w+)", src)
    launched = {w for w in launches if w in kernels}
    for line in re.findall(r"auto kernel = [^;]*;", src):
        launched |= set(re.findall(r"\bk_\w+", line))
    assert launched and launched <= {k for k, b in kernels.items() if "pdl_wait()" in b}
