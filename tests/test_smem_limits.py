"""A kernel's limit of dynamic shared memory holds for the whole process.  It
is set through smem_limit (csrc/ph0_common.cuh), whose size is a template
argument: a size that depends on the call, which another thread's call could
lower before the launch, does not compile."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_02527_gb300", "csrc")


def test_limits_are_compile_time_sizes():
    found = {}
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = open(os.path.join(CSRC, f)).read()
        found[f] = re.findall(r"cudaFuncAttributeMaxDynamicSharedMemorySize,\s*([^;]*);", text)
    assert {f: sizes for f, sizes in found.items() if sizes} == {"ph0_common.cuh": ["int(kBytes))"]}
