"""Table kernel at the sizes where its blocks, masks and scans end: tables bit-exact against the oracle."""
import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import synth

pytestmark = pytest.mark.gpu

# (documents, slots): one 1024-slot block and its neighbours, mask words of 32 and 64 slots, several passes of the document
# scan, and both sides of the limits (4096 documents, 65536 slots) up to which one launch does everything
SIZES = [(1, 1), (1, 31), (2, 32), (3, 33), (5, 63), (5, 64), (7, 65), (40, 1023), (40, 1024), (41, 1025), (1023, 2049), (1024, 2048),
         (1025, 3000), (4096, 9000), (4097, 9000), (9, 65535), (9, 65536), (9, 65537)]


@pytest.mark.parametrize("misaligned", [0, 1])
@pytest.mark.parametrize("docs,slots", SIZES)
def test_tables_at_block_edges(docs, slots, misaligned):
    from oracle import capi
    from paper_2604_26209_b200 import binding as B
    rng = np.random.default_rng([docs, slots])
    cut = np.sort(rng.integers(0, slots + 1, size=docs - 1))          # equal cuts: documents without slots
    cnt = np.diff(np.concatenate([[0], cut, [slots]])).astype(np.int32)
    L = rng.integers(0, 3000, size=docs).astype(np.int32)
    depth = rng.integers(0, 4, size=slots).astype(np.int32)
    alive = (rng.random(slots) < 0.6).astype(np.uint8) * rng.integers(1, 256, size=slots).astype(np.uint8)
    alive[-1] = 1
    g = synth.Geom(Hq=2, Hkv=1, D=64, rope_theta=10000.0, sm_scale=0.125, suffix_cap=4)
    m = B.MetaTables.alloc(g, docs, slots, int(L.sum()))
    dev = lambda a: torch.from_numpy(a).cuda()                        # noqa: E731
    buf = torch.zeros(slots + misaligned, dtype=torch.uint8, device="cuda")
    buf[misaligned:] = dev(alive)
    B.hpd_build_meta(g, docs, slots, dev(L), dev(cnt), dev(depth), buf[misaligned:], 5, m)
    torch.cuda.synchronize()
    want = capi.build_meta(L, cnt, depth, alive, g.suffix_cap, 5)
    assert int(m.n_active.item()) == want.n_active
    for name in capi.Meta.TABLES:
        w = getattr(want, name)
        assert np.array_equal(getattr(m, name).cpu().numpy()[:len(w)], w), name


@pytest.mark.parametrize("docs", [3, 1500])
@pytest.mark.parametrize("wrong", [-1, -40, -2**31, 2**31 - 1])
def test_counts_outside_the_slots_stay_inside_the_tables(docs, wrong):
    """A count no document can have is taken as 0 or as all slots: first slots ascend, every row range lies inside the rows."""
    from paper_2604_26209_b200 import binding as B
    slots = 2 * docs
    cnt = np.full(docs, 2, np.int32)
    cnt[docs // 2] = wrong
    g = synth.Geom(Hq=2, Hkv=1, D=64, rope_theta=10000.0, sm_scale=0.125, suffix_cap=4)
    m = B.MetaTables.alloc(g, docs, slots, docs)
    dev = lambda a: torch.from_numpy(a).cuda()                        # noqa: E731
    B.hpd_build_meta(g, docs, slots, dev(np.ones(docs, np.int32)), dev(cnt), dev(np.zeros(slots, np.int32)), dev(np.ones(slots, np.uint8)), 0, m)
    torch.cuda.synchronize()
    first = np.concatenate([[0], np.cumsum(np.clip(cnt, 0, slots))])
    assert int(m.n_active.item()) == slots
    assert np.array_equal(m.doc_slot_start.cpu().numpy()[:docs + 1], first)
    assert np.array_equal(m.doc_active_start.cpu().numpy()[:docs + 1], np.concatenate([np.minimum(first[:-1], slots), [slots]]))


@pytest.mark.parametrize("offset", [2, 7, 8, 15])
@pytest.mark.parametrize("docs,slots", [(1, 1), (2, 17), (3, 33), (5, 64), (40, 1023), (9, 65536)])
def test_live_flags_at_any_address(docs, slots, offset):
    test_tables_at_block_edges(docs, slots, offset)
