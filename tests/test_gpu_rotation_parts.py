"""Rotation of few rows, where several CTAs share a pair of rows: the row counts at which the number of CTAs to a pair changes (up to five
batches of chunks at 32 + 8 heads of 128), both with and without the append, and a step with retired rows."""
import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import synth

pytestmark = pytest.mark.gpu


def _edges():
    """Rows around the steps of floor(resident CTAs / row pairs) for 148 SMs of six or eight CTAs."""
    out = {1, 2, 3}
    for wave in (6 * 148, 8 * 148):
        for parts in (2, 3, 4, 5):
            out |= {2 * (wave // parts) - 1, 2 * (wave // parts) + 1}
    return sorted(out)


@pytest.mark.parametrize("rows", _edges())
@pytest.mark.parametrize("Hq,Hkv,D", [(32, 8, 128), (8, 1, 64), (5, 5, 128)])
def test_rows_shared_by_ctas(rows, Hq, Hkv, D):
    from oracle import capi
    from paper_2604_26209_b200 import binding as B, runtime
    g = synth.Geom(Hq=Hq, Hkv=Hkv, D=D, rope_theta=500000.0, sm_scale=0.125, suffix_cap=2)
    gen = torch.Generator(device="cuda").manual_seed(rows)
    q, k, v = (torch.randn(rows, h, D, device="cuda", generator=gen).to(torch.bfloat16) for h in (Hq, Hkv, Hkv))
    live = max(1, rows - 2)                                           # the last rows are not there
    pos = torch.arange(rows, dtype=torch.int32, device="cuda") * 3
    off, length = 2 * torch.arange(rows, dtype=torch.int32, device="cuda"), torch.arange(rows, dtype=torch.int32, device="cuda") % 2
    n, status = torch.tensor([live], dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    cache = [torch.zeros(2 * rows, Hkv, D, dtype=torch.bfloat16, device="cuda") for _ in range(4)]
    q1, k1, q2, k2 = q.clone(), k.clone(), q.clone(), k.clone()
    B.hpd_rope(g, rows, n, pos, q1, k1)
    B.hpd_kv_append(g, rows, rows, n, off, length, k1, v, cache[0], cache[1], status)
    B.hpd_rope_append(g, rows, rows, n, pos, off, length, q2, k2, v, cache[2], cache[3], status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert torch.equal(q1, q2) and torch.equal(k1, k2) and torch.equal(cache[0], cache[2]) and torch.equal(cache[1], cache[3])
    assert torch.equal(q1[live:], q[live:]) and torch.equal(k1[live:], k[live:])
    for got, x in ((q1, q), (k1, k)):
        for r in sorted({0, live // 2, live - 1}):
            exact = capi.rope(synth.bf16_bits_to_f32(runtime.bits_of(x[r:r + 1]))[0], 3 * r, g.rope_theta)
            row = synth.bf16_bits_to_f32(runtime.bits_of(got[r:r + 1]))[0]
            assert np.all(np.abs(row - exact) <= 2.0 ** -8 * np.abs(exact) + 1e-5)       # half a bf16 step, and the fp32 rotation
