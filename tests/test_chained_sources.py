"""Kernels that start before their predecessor in the stream has ended must not promise that nobody writes their operands."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_26209_b200", "csrc")


WAIT, LET_IN = "await_predecessors();", "start_dependents();"


def _chained():
    """{name: (parameter list, code)} of every kernel that waits for its predecessors itself."""
    text = "\n".join(open(f).read() for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))))
    found = {}
    for kernel in re.split(r"(?=__global__)", text)[1:]:
        name, params = re.match(r"__global__[^;{]*?\b(\w+_kernel)\((.*?)\)\s*\{", kernel, re.S).groups()
        if WAIT in kernel:
            found[name] = params, re.sub(r"//[^\n]*", "", kernel)
    return found


def test_chained_kernels_have_no_restrict_parameters():
    kernels = _chained()
    assert set(kernels) == {"advance_kernel", "hpd_attn_tc_kernel", "hpd_merge_kernel", "meta_step_kernel", "prefill_meta_kernel", "rope_kernel"}
    for name, (params, _) in kernels.items():
        assert "__restrict__" not in params, f"{name}: a predecessor may still write what a __restrict__ parameter points to"


def test_only_the_merge_kernel_ends_blocks_before_its_wait_and_never_block_0():
    for name, (_, code) in _chained().items():
        before = code[: code.index(WAIT)]
        if name == "hpd_merge_kernel":
            assert re.findall(r"if \(([^;{]*)\) return;", before) == ["!any_split && blockIdx.x > 0"] and before.count("return;") == 1
        else:
            assert "return;" not in before, name


def test_attention_lets_the_merge_kernel_in_after_its_own_wait():
    """The merge kernel reads the plan before it waits: the attention must have seen the plan's kernel end by then, in every block."""
    code = _chained()["hpd_attn_tc_kernel"][1]
    assert code.count(LET_IN) == 1
    assert code.rindex(WAIT) < code.index(LET_IN)
    # nothing but the refusal of a misaligned segment, which waits itself, leaves the kernel in front of it
    assert code[: code.index(LET_IN)].count("return;") == 1


def test_merge_and_rotation_let_their_successors_in_after_their_wait():
    for name in ("hpd_merge_kernel", "rope_kernel"):
        code = _chained()[name][1]
        assert code.count(LET_IN) == 1 and code.index(WAIT) < code.index(LET_IN), name
