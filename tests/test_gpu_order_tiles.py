"""Position-order decode where its K and V producers change over: packed cached tokens just below, at and past whole tiles of 64 and past the
rings' stages, units without cached tokens, and more units than pipelines (each producer then runs ahead into the next unit)."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import synth
from tests.test_gpu_posorder import _oracle
from tests.util import err_stats

pytestmark = pytest.mark.gpu

GEOMS = {"d128": dict(Hq=32, Hkv=8, D=128, theta=500000.0), "d64": dict(Hq=8, Hkv=2, D=64, theta=1e4)}
# name: prompt lengths, slots per group, depths of the slots (repeated), live flags (repeated)
CASES = {
    "63_columns": ([70], [63], [0], [1]), "64_columns": ([70], [64], [0], [1]), "65_columns": ([1], [65], [0], [1]),
    "one_live_retired_empty": ([130], [40], [0], [0, 0, 1]),
    "past_the_rings": ([64], [96], [6, 7, 5], [1, 1, 0]),
    "no_prompt": ([0, 0], [33, 5], [3], [1]),
    "many_units": ([40 + 13 * (i % 7) for i in range(90)], [3 + i % 5 for i in range(90)], [0, 1, 7], [1, 0, 1]),
}


@pytest.mark.parametrize("geom", list(GEOMS))
@pytest.mark.parametrize("name", list(CASES))
def test_producers_at_tile_edges(name, geom):
    from paper_2604_26209_b200 import runtime as rt
    lens, cnt, depth, alive = CASES[name]
    s = synth.config_skeleton(name, **GEOMS[geom], k_max=8, prompt_lens=lens, branch_cnts=cnt, key_len_hi=2, seed=11)
    n = s.n_slots
    s = replace(s, slot_depth=np.resize(depth, n).astype(np.int32), slot_alive=np.resize(alive, n).astype(np.uint8))
    tb = synth.make_tensors(s)
    meta, _, want = _oracle(s, tb)
    db = rt.DeviceBatch(s, tb)
    db.build_meta()
    act = meta.active_slot[: meta.n_active]
    db.set_step_inputs(tb["q"][act], tb["k_new"][act], tb["v_new"][act])
    db.rope_append()
    db.attn(True)
    torch.cuda.synchronize()
    assert db.status() == 0
    o = synth.bf16_bits_to_f32(rt.bits_of(db.o))[: meta.n_active]
    mx, mean = err_stats(o, want.o)
    assert mx <= 2e-2 and mean <= 2e-3, (mx, mean)                    # the tolerance of the mode's other tests: bf16 in and out
    assert np.max(np.abs(db.lse.cpu().numpy()[: meta.n_active] - want.lse)) <= 2e-2
