"""Whole steps around the unit counts where the attention kernel's list changes its way over the SMs (148 SMs, two pipelines each,
four rounds) and the rotary kernel's two-row blocks end, against the oracle (bars of tests/test_gpu_parity.py)."""
import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import synth
from tests.util import err_stats, oracle_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("units", [1, 2, 3, 147, 148, 149, 295, 296, 297, 1183, 1184, 1185])
def test_step_at_unit_counts(units):
    from paper_2604_26209_b200 import runtime
    s = synth.config_custom("units", Hq=2, Hkv=1, D=64, theta=10000.0, cap=4, prefix_lens=[(41 * i) % 150 for i in range(units)],
                            branch_cnts=[1] * units, depth_hi=4, seed=units, alive_frac=1.0)
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
    assert n == meta.n_active == units and db.status() == 0
    mx, mean = err_stats(synth.bf16_bits_to_f32(runtime.bits_of(db.o))[:n], want.o)
    assert mx <= 2e-2 and mean <= 2e-3, (mx, mean)
    assert np.max(np.abs(db.lse.cpu().numpy()[:n] - want.lse)) <= 2e-2
