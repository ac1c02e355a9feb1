"""End of a step around the sizes where its launch changes (one block of 1024 rows, several passes of it, many blocks)."""
import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [0, 1, 1023, 1024, 1025, 8191, 8192, 8193, 20000])
@pytest.mark.parametrize("idle", [0, 7])          # rows of the tables beyond n_active
def test_advance_at_block_edges(rows, idle):
    from paper_2604_26209_b200 import binding as B
    rng = np.random.default_rng([rows, idle])
    n, cap = rows + idle, 5
    g = synth.Geom(Hq=2, Hkv=1, D=64, rope_theta=10000.0, sm_scale=0.125, suffix_cap=cap)
    slot = rng.permutation(n).astype(np.int32)
    depth, token = rng.integers(0, cap + 1, size=n).astype(np.int32), rng.integers(0, 3, size=n).astype(np.int32)
    alive = np.ones(n, np.uint8)
    d, a = depth.copy(), alive.copy()
    d[slot[:rows]] = np.minimum(d[slot[:rows]] + 1, cap)
    a[slot[:rows]] = (token[:rows] != 1) & (d[slot[:rows]] < cap)
    dev = lambda x: torch.from_numpy(x if len(x) else np.zeros(1, x.dtype)).cuda()          # noqa: E731
    gd, ga = dev(depth), dev(alive)
    count = torch.full((1,), 77, dtype=torch.int32, device="cuda")
    B.hpd_advance(g, n, dev(np.array([rows], np.int32)), dev(slot), dev(token), 1, gd, ga, count)
    torch.cuda.synchronize()
    assert int(count.item()) == int(a[slot[:rows]].sum())
    assert np.array_equal(gd.cpu().numpy()[:n], d) and np.array_equal(ga.cpu().numpy()[:n], a)


@pytest.mark.parametrize("rows", [2047, 2048, 2049, 4095, 4096, 4097, 6145])
def test_advance_at_pass_edges(rows):
    test_advance_at_block_edges(rows, 0)
    test_advance_at_block_edges(rows, 5000)          # idle entries past the one-block limit
