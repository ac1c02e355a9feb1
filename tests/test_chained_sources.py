"""Kernels that start before their predecessor in the stream has ended must not promise that nobody writes their operands."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_26209_b200", "csrc")


def _chained():
    """{name: parameter list} of every kernel that waits for its predecessors itself."""
    text = "\n".join(open(f).read() for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))))
    found = {}
    for kernel in re.split(r"(?=__global__)", text)[1:]:
        name, params = re.match(r"__global__[^;{]*?\b(\w+_kernel)\((.*?)\)\s*\{", kernel, re.S).groups()
        if "await_predecessors();" in kernel:
            found[name] = params
    return found


def test_chained_kernels_have_no_restrict_parameters():
    kernels = _chained()
    assert set(kernels) == {"advance_kernel", "hpd_attn_tc_kernel", "hpd_merge_kernel", "meta_step_kernel", "prefill_meta_kernel", "rope_kernel"}
    for name, params in kernels.items():
        assert "__restrict__" not in params, f"{name}: a predecessor may still write what a __restrict__ parameter points to"
