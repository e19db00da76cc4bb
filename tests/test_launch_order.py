"""Order of the dependents' launch and the tensor-memory allocation in every kernel source (no GPU needed): a kernel that lets
its dependents start before its own allocation is granted can be locked out of tensor memory by a dependent that waits for it."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_20386_b200", "csrc")


def kernels():
    """(name, body) of every __global__ function, comments removed."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?(ptq_\w+)\s*\(", text):
            start = text.index("{", text.index(")", m.end()))
            depth, i = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            out.append((m.group(1), text[start:i]))
    return out


ALLOCATING = [(n, b) for n, b in kernels() if "tmem_alloc" in b and "griddep_launch_dependents" in b]


def test_the_kernels_are_found():
    assert {"ptq_small_kernel", "ptq_short_k_kernel", "ptq_gemm_dequant_kernel", "ptq_gemm_dequant_panel_kernel",
            "ptq_gemm_dequant_resident_kernel"} <= {n for n, _ in ALLOCATING}


@pytest.mark.parametrize("name,body", ALLOCATING, ids=[n for n, _ in ALLOCATING])
def test_dependents_are_launched_behind_the_allocation(name, body):
    alloc = max(m.start() for m in re.finditer(r"tmem_alloc\w*\(", body))
    launch = body.index("griddep_launch_dependents()")
    assert alloc < launch and "__syncthreads()" in body[alloc:launch], name
