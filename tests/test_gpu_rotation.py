"""Rotation and append at the row counts where their grids stop fitting the GPU at once (two rows per CTA, eight CTAs an SM for the
rotation alone, six with the append) and the next kernel is not let in early any more."""
import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_sm", [6, 8])
@pytest.mark.parametrize("rows_off", [-1, 0, 1])
def test_rotation_at_wave_edges(per_sm, rows_off):
    from oracle import capi
    from paper_2604_26209_b200 import binding as B, runtime
    rows = 2 * per_sm * torch.cuda.get_device_properties(0).multi_processor_count + rows_off
    g = synth.Geom(Hq=2, Hkv=1, D=64, rope_theta=10000.0, sm_scale=0.125, suffix_cap=2)
    gen = torch.Generator(device="cuda").manual_seed(rows)
    q, k, v = (torch.randn(rows, h, 64, device="cuda", generator=gen).to(torch.bfloat16) for h in (2, 1, 1))
    pos = torch.arange(rows, dtype=torch.int32, device="cuda")
    off, length, n, status = 2 * pos, pos % 2, torch.tensor([rows], dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    want = [np.stack([capi.rope(x, r, g.rope_theta) for r, x in enumerate(synth.bf16_bits_to_f32(runtime.bits_of(t)))]) for t in (q, k)]
    cache = [torch.zeros(2 * rows, 1, 64, dtype=torch.bfloat16, device="cuda") for _ in range(4)]
    q2, k2 = q.clone(), k.clone()
    B.hpd_rope(g, rows, n, pos, q, k)
    B.hpd_kv_append(g, rows, rows, n, off, length, k, v, cache[0], cache[1], status)
    B.hpd_rope_append(g, rows, rows, n, pos, off, length, q2, k2, v, cache[2], cache[3], status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for got, exact in zip((q, k), want):
        got = synth.bf16_bits_to_f32(runtime.bits_of(got))
        assert np.all(np.abs(got - exact) <= 2.0 ** -8 * np.abs(exact) + 1e-5)           # half a bf16 step, and the fp32 rotation
    assert torch.equal(q, q2) and torch.equal(k, k2) and torch.equal(cache[0], cache[2]) and torch.equal(cache[1], cache[3])
