"""Kernels launched while the kernel before them still runs (they call
depend_wait) read its output: their loads must be ordinary ones.  __ldg and const
__restrict__ parameters promise memory that nothing writes during the kernel, and
such loads may be moved above the wait.  A wrong load would be a race on the GPU,
so it is looked for in the source."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2609_32259_gb300", "csrc")


def _code(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    return re.sub(r"/\*.*?\*/", "", text, flags=re.S)


def _kernels(text):
    """(name, parameters and body) of every __global__ function."""
    parts = re.split(r"__global__", text)[1:]
    return [(re.search(r"(\w+)\s*\((?!\()[^()]*(?:const|float|int)", p).group(1), p) for p in parts]


# fold_b_kernel reads nothing that the kernel before it writes, and that kernel is
# launched after everything before it has ended
EXEMPT = {"fold_b_kernel"}


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_dependent_kernels_make_ordinary_loads(name):
    text = _code(name)
    if "depend_wait" not in text:
        return
    if name != "hf_fold.cu":  # device functions of these files serve dependent kernels
        assert "__ldg(" not in text and "ld.global.nc" not in text
    for kernel, body in _kernels(text):
        if "depend_wait" in body and kernel not in EXEMPT:
            signature = body[:body.index("{")]
            assert not re.search(r"const[^,]*\*\s*__restrict__", signature), kernel
