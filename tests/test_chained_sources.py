"""Kernels that start before their predecessor in the stream has ended must not promise that nobody writes their operands."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_26209_b200", "csrc")


def _chained():
    """(name, parameter list) of every kernel handed to launch_chained."""
    text = "\n".join(open(f).read() for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))))
    found = []
    for name in sorted(set(re.findall(r"launch_chained\((?:[^,]*\? *)?(\w+)", text))):
        m = re.search(r"__global__[^;{]*?\b" + name + r"\((.*?)\)\s*\{.*?await_predecessors\(\);", text, re.S)
        assert m, f"{name}: no definition with a wait"
        found.append((name, m.group(1)))
    return found


def test_chained_kernels_have_no_restrict_parameters():
    kernels = _chained()
    assert [k[0] for k in kernels] == ["advance_kernel", "hpd_attn_tc_kernel", "hpd_merge_kernel", "meta_step_kernel", "prefill_meta_kernel",
                                       "rope_kernel"]
    for name, params in kernels:
        assert "__restrict__" not in params, f"{name}: a predecessor may still write what a __restrict__ parameter points to"
