"""The FP64 level kernels are set up while the kernel before them runs, and the
batched kernel writes what it reads: no read-only load in their sources but
the FP32 one of ld_level."""
import os
import re

from paper_1807_00370_gb300 import build

SHARED = ("cr_core.cuh", "cr_core64.cuh", "cr_split.cuh", "cr_tail.cu", "cr_batch.cuh")


def _code(name):
    text = open(os.path.join(build.CSRC, name)).read()
    return re.sub(r"//.*", "", text)


def test_no_read_only_loads_in_the_fp64_levels():
    for name in SHARED:
        code = _code(name)
        assert "__ldg" not in code and "ld.global.nc" not in code and "__restrict__" not in code, name
    uses = [line for line in _code("cr_device.cuh").splitlines() if "__ldg" in line]
    assert len(uses) == 1 and "float2 ld_level(const float2" in uses[0]
