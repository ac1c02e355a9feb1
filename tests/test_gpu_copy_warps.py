"""Whole decode steps through the kernel with copy warps, at D = 128 and 64: one unit an SM (the copy warps of the idle pipeline help) up to the
last SM and past it, several units a pipeline, and documents so uneven that the units are not those that the host expects."""
import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import synth
from tests.util import copy_warps_rule, err_stats, oracle_step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    return copy_warps_rule(str(tmp_path_factory.mktemp("rule")))


def _even(docs, branches, tokens):
    return [max(0, tokens + (i % 5) - 2) for i in range(docs)], [branches] * docs


# name: (Hq, Hkv, D), prefix lengths and branches of the documents, which kernel, units against SMs
CASES = {
    "one_before_the_last_sm": ((4, 1, 128), *_even(147, 24, 40), True, "<="), "the_last_sm": ((4, 1, 128), *_even(148, 24, 40), True, "<="),
    "one_past_the_last_sm": ((4, 1, 128), *_even(149, 24, 40), False, ">"), "many_units_d128": ((8, 8, 128), *_even(18, 150, 70), True, ">"),
    "many_units_d64": ((8, 4, 64), *_even(36, 90, 70), True, ">"), "split_one_an_sm": ((8, 8, 128), *_even(3, 128, 1600), True, "<="),
    "split_several_an_sm": ((8, 8, 128), *_even(18, 48, 900), True, ">"),
    "more_units_than_expected": ((4, 1, 128), [60] * 70, [33] * 60 + [200] * 10, True, ">"),
    "long_document_among_short": ((8, 8, 128), [1200] + [30] * 17, [48] * 18, True, ">"),
    "fewer_units_than_expected": ((8, 8, 128), [4000] + [444] * 9, [128] * 10, True, "<="),
    "many_short_units": ((4, 1, 128), *_even(120, 160, 20), True, ">"),
    "no_prefix": ((8, 2, 128), [0] * 12, [40] * 12, True, "<="),
}


@pytest.mark.parametrize("name", list(CASES))
def test_step_with_copy_warps(rule, name):
    from paper_2604_26209_b200 import runtime
    (Hq, Hkv, D), lens, cnts, pay, side = CASES[name]
    s = synth.config_custom(name, Hq=Hq, Hkv=Hkv, D=D, theta=10000.0, cap=7, prefix_lens=lens, branch_cnts=cnts, depth_hi=7, seed=len(lens),
                            alive_frac=1.0)
    tb = synth.make_tensors(s)
    meta, want = oracle_step(s, tb)
    db = runtime.DeviceBatch(s, tb)
    db.build_meta()
    n = db.tables()["n_active"]
    act = db.tables()["active_slot"][:n]
    db.set_step_inputs(tb["q"][act], tb["k_new"][act], tb["v_new"][act])
    db.rope_append()
    db.attn(True)
    torch.cuda.synchronize()
    assert n == meta.n_active == sum(cnts) and db.status() == 0
    header = db.meta.workspace.cpu().numpy().view(np.int32)           # work items, ..., capacities (WsHeader)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert rule(len(lens), sum(cnts), sum(lens), Hq // Hkv, Hkv, D, sm, int(header[5]), int(header[6]))[0] == pay
    assert (int(header[0]) * Hkv <= sm) == (side == "<=")
    mx, mean = err_stats(synth.bf16_bits_to_f32(runtime.bits_of(db.o))[:n], want.o)
    assert mx <= 2e-2 and mean <= 2e-3, (mx, mean)                    # the bars of tests/test_gpu_parity.py
    assert np.max(np.abs(db.lse.cpu().numpy()[:n] - want.lse)) <= 2e-2
