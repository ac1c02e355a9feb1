"""Rotation of few rows, where several CTAs share a pair of rows, at the row counts where the number of CTAs to a pair changes, with and without
the append and with retired rows: D = 128 and 64, one batch of chunks (never shared), as many as a thread holds, and more (a thread then reads
and writes in several passes, of q and k and of v)."""
import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import synth

pytestmark = pytest.mark.gpu

THREADS, HELD, HELD_V = 128, 5, 2                                     # of a CTA; chunk pairs and value pieces that a thread holds at once
RESIDENT = {"fused": 6, "alone": 8}                                   # CTAs of an SM
# (Hq, Hkv, D): batches of chunk pairs of two rows
GEOMS = {(32, 8, 128): 5, (5, 5, 128): 2, (32, 8, 64): 3, (32, 32, 128): 8, (64, 64, 128): 16, (64, 64, 64): 8, (8, 1, 64): 1}


SHARING = [(g, p) for g, b in GEOMS.items() for p in sorted({2, 3, 4, b}) if p <= max(2, b) and p > 1]


@pytest.mark.parametrize("side", ["last_shared_by_so_many", "first_shared_by_fewer"])
@pytest.mark.parametrize("kernel", list(RESIDENT))
@pytest.mark.parametrize("geom,parts", SHARING, ids=lambda x: "-".join(map(str, x)) if isinstance(x, tuple) else str(x))
def test_rows_shared_by_ctas(geom, parts, kernel, side):
    Hq, Hkv, D = geom
    batches = -(-2 * (Hq + Hkv) * (D // 16) // THREADS)
    assert batches == GEOMS[geom]
    wave = RESIDENT[kernel] * torch.cuda.get_device_properties(0).multi_processor_count
    pairs = wave // parts + (side == "first_shared_by_fewer")
    shared = min(wave // pairs, batches)                              # the launch's rule
    assert shared == 1 if batches == 1 else shared >= parts if side == "last_shared_by_so_many" else shared < parts
    _check(Hq, Hkv, D, 2 * pairs - 1)                                 # a row without a partner at the end


@pytest.mark.parametrize("rows", [1, 2, 3])
@pytest.mark.parametrize("geom", list(GEOMS), ids=lambda g: "-".join(map(str, g)))
def test_one_and_two_pairs(geom, rows):
    _check(*geom, rows)


def test_the_sizes_take_every_path():
    """Several passes of q and k, and of v, among CTAs that share: more batches to a CTA than its threads hold."""
    passes = {g: [-(-b // p) for p in (2, 3)] for g, b in GEOMS.items()}
    assert all(n > HELD for n in passes[64, 64, 128]) and all(n <= HELD for n in passes[32, 32, 128])
    v_batches = {(q, k, d): 2 * k * d // 8 / THREADS for q, k, d in GEOMS}
    assert v_batches[32, 32, 128] / 3 > HELD_V and v_batches[32, 8, 128] / 2 <= HELD_V


def _check(Hq, Hkv, D, rows):
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
    # the cache: v and the rotated k at each live row's place, nothing anywhere else
    want = torch.zeros(2, 2 * rows, Hkv, D, dtype=torch.bfloat16, device="cuda")
    at = (off + length)[:live].long()
    want[0, at], want[1, at] = k1[:live], v[:live]
    assert torch.equal(cache[2], want[0]) and torch.equal(cache[3], want[1])
    for got, x in ((q1, q), (k1, k)):
        for r in sorted({0, live // 2, live - 1}):
            exact = capi.rope(synth.bf16_bits_to_f32(runtime.bits_of(x[r:r + 1]))[0], 3 * r, g.rope_theta)
            row = synth.bf16_bits_to_f32(runtime.bits_of(got[r:r + 1]))[0]
            assert np.all(np.abs(row - exact) <= 2.0 ** -8 * np.abs(exact) + 1e-5)       # half a bf16 step, and the fp32 rotation
        # all rows: the same rotation by torch, in 64 bits
        half = D // 2
        ang = (pos[:live].double()[:, None] * g.rope_theta ** (-2.0 * torch.arange(half, device="cuda", dtype=torch.float64) / D))[:, None, :]
        a, b = x[:live, :, :half].double(), x[:live, :, half:].double()
        ref = torch.cat([a * ang.cos() - b * ang.sin(), b * ang.cos() + a * ang.sin()], -1)
        assert bool(((got[:live].double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-5).all())
