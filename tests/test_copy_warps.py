"""The rule that gives a decode launch copy warps: by the branches and keys of its units and by how many of them an SM gets, not by documents."""
import pytest

from tests.util import copy_warps_rule

SM, CAP = 148, 1 << 30


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    return copy_warps_rule(str(tmp_path_factory.mktemp("rule")))


# documents, branches of each, tokens of each, G, Hkv, D -> units, copy warps
@pytest.mark.parametrize("docs,branches,tokens,G,Hkv,D,units,pay", [
    # several units an SM: many branches per document, or documents split to fill the SMs (each measured 2 to 8 % slower with copy warps)
    (4, 480, 128, 4, 8, 128, 480, False), (4, 480, 8192, 4, 8, 128, 480, False), (8, 96, 128, 4, 8, 128, 192, False),
    (1, 96, 8192, 4, 8, 128, 192, False), (8, 24, 2048, 4, 8, 128, 256, False), (18, 48, 1000, 8, 4, 128, 216, False),
    (18, 48, 4000, 1, 8, 128, 288, False), (148, 48, 4000, 4, 1, 64, 296, False),
    # one unit an SM of few branches
    (4, 4, 512, 4, 8, 128, 32, False), (4, 48, 200, 8, 4, 128, 48, False), (64, 8, 1000, 4, 1, 64, 128, False),
    # one unit an SM of many, at its edges
    (4, 24, 512, 4, 8, 128, 32, True), (1, 480, 512, 4, 8, 128, 120, True), (1, 24, 8192, 4, 8, 128, 128, True), (148, 24, 100, 4, 1, 128, 148, True),
    (149, 24, 100, 4, 1, 128, 149, False), (4, 21, 512, 4, 8, 128, 32, False), (4, 22, 512, 4, 8, 128, 32, True),
    # many branches against few keys
    (18, 48, 1000, 1, 8, 128, 288, True), (18, 200, 200, 1, 8, 128, 288, True), (35, 56, 1500, 2, 4, 64, 280, True), (18, 64, 1500, 1, 8, 128, 288, False),
    # many short units of 32 branches
    (8, 480, 512, 4, 8, 128, 960, True), (8, 480, 513, 4, 8, 128, 960, False), (5, 448, 128, 4, 8, 128, 560, False), (5, 480, 128, 4, 8, 128, 600, True),
    # one row, one document, no prefix
    (1, 1, 0, 1, 1, 64, 1, False),
])
def test_units_decide(rule, docs, branches, tokens, G, Hkv, D, units, pay):
    assert rule(docs, docs * branches, docs * tokens, G, Hkv, D, SM, CAP, CAP) == (pay, units)


def test_workspace_limits_the_split(rule):
    """48 branches of 4 documents of 4000 tokens: eight chunks of 512 keys, or four where eight chunks' partial rows do not fit."""
    assert rule(4, 192, 16000, 1, 8, 128, SM, CAP, CAP) == (True, 256)
    assert rule(4, 192, 16000, 1, 8, 128, SM, CAP, 192 * 8 - 1) == (True, 128)
    assert rule(4, 192, 16000, 1, 8, 128, SM, 4 * 2, CAP) == (True, 64)


def test_largest_sizes_do_not_overflow(rule):
    big = 2 ** 31 - 1
    assert rule(1, big, big, 1, 1, 128, SM, big, big)[1] == (big - 1) // 128 + 1
    assert rule(big, big, big, 8, 4096, 64, SM, big, big) == (False, big * 4096)


@pytest.mark.parametrize("docs,branches,tokens,G,Hkv", [(1, 96, 128, 4, 8), (4, 96, 300, 4, 8), (1, 6144, 128, 4, 8), (18, 200, 200, 1, 8)])
def test_calls_without_the_steps_tokens_have_nothing_to_copy(rule, docs, branches, tokens, G, Hkv):
    """A block's pass over all rows below it (measured 5 to 18 % slower with copy warps)."""
    assert rule(docs, docs * branches, docs * tokens, G, Hkv, 128, SM, CAP, CAP)[0]
    assert not rule(docs, docs * branches, docs * tokens, G, Hkv, 128, SM, CAP, CAP, new_tokens=0)[0]
