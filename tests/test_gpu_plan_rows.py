"""A work item names its document's first row, so that a unit's tables can be asked for with it: the rows in the lists of both table paths and of
the first inference step, and attention calls whose row tables were moved after the list was made (the tables passed decide)."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import synth

pytestmark = pytest.mark.gpu

dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()                                     # noqa: E731


def _items(workspace):
    words = workspace.cpu().numpy()[: workspace.numel() // 4 * 4].view(np.int32)
    return words[64: 64 + 8 * words[0]].reshape(-1, 8)                # WorkItems behind the 256 bytes of the WsHeader


# name: documents' tokens, branches (both repeated over the documents), documents, share of live branches
LISTS = {"row_blocks": ([40, 0, 300], [70, 0, 33, 1, 200], 5, 0.8), "split": ([3000, 900, 2], [5, 3], 4, 1.0), "one": ([7], [1], 1, 1.0),
         "three_kernels": ([5, 900, 0], [1, 40, 0, 2], 4200, 0.6)}


@pytest.mark.parametrize("name", list(LISTS))
def test_items_name_their_documents_first_row(name):
    from paper_2604_26209_b200 import binding as B
    lens, cnts, docs, share = LISTS[name]
    L, cnt = np.resize(lens, docs).astype(np.int32), np.resize(cnts, docs).astype(np.int32)
    n = int(cnt.sum())
    rng = np.random.default_rng(docs)
    alive = (rng.random(n) < share).astype(np.uint8)
    alive[0] = 1
    g = synth.Geom(Hq=4, Hkv=1, D=64, rope_theta=10000.0, sm_scale=0.125, suffix_cap=4)
    m = B.MetaTables.alloc(g, docs, n, int(L.sum()))
    B.hpd_build_meta(g, docs, n, dev(L), dev(cnt), dev(np.zeros(n, np.int32)), dev(alive), 0, m)
    torch.cuda.synchronize()
    items, first = _items(m.workspace), m.doc_active_start.cpu().numpy()
    rows = np.diff(np.concatenate([[0], np.cumsum(alive)])[np.concatenate([[0], np.cumsum(cnt)])])
    assert np.array_equal(np.diff(first), rows) and np.array_equal(items[:, 7], first[items[:, 0]])
    # every live row is in the list, and no row of another document
    assert set(items[:, 0]) == set(np.flatnonzero(rows)) and np.all(items[:, 4] + items[:, 5] <= rows[items[:, 0]])


def test_first_step_items_name_their_prompts_first_token():
    from paper_2604_26209_b200 import binding as B
    L = np.array([300, 0, 33, 32, 1, 700], np.int32)
    g = synth.Geom(Hq=4, Hkv=1, D=64, rope_theta=10000.0, sm_scale=0.125, suffix_cap=4)
    t = B.PrefillTables.alloc(g, len(L), int(L.sum()))
    B.hpd_prefill_meta(g, len(L), 0, int(L.sum()), dev(L), dev(np.zeros(len(L), np.int32)), dev(np.zeros(1, np.int32)), 0, t)
    torch.cuda.synchronize()
    items = _items(t.workspace)
    assert len(items) == sum((l + 31) // 32 for l in L)
    assert np.array_equal(items[:, 7], t.doc_kv_start.cpu().numpy()[items[:, 0]])


MOVED = 37
# name: (Hq, Hkv, D), documents' tokens, branches, position order
CALLS = {"own": ((8, 2, 128), [200, 3, 90], [9, 70, 1], False, 60), "copy_warps": ((8, 2, 128), [100, 700], [40, 64], False, 5),
         "copy_warps_d64": ((4, 4, 64), [60], [50], False, 30), "split": ((8, 2, 128), [3000, 2000], [4, 30], False, 2),
         "order": ((8, 2, 128), [90, 400], [40, 90], True, 40), "order_split": ((8, 2, 128), [2500], [60], True, 2)}


@pytest.mark.parametrize("name", list(CALLS))
def test_tables_moved_after_the_list_was_made(name):
    """The same rows 37 places further in every row table, with the list of the tables as they were: the same output, 37 places further."""
    from paper_2604_26209_b200 import binding as B
    (Hq, Hkv, D), lens, cnts, order, docs = CALLS[name]
    L, cnt = np.resize(lens, docs + 1).astype(np.int32), np.resize(cnts, docs + 1).astype(np.int32)
    cnt[-1] = 0                                                       # no rows: the merge passes over the rows in front, which are given to it
    n, T, cap = int(cnt.sum()), int(L.sum()), 5
    g = synth.Geom(Hq=Hq, Hkv=Hkv, D=D, rope_theta=10000.0, sm_scale=D ** -0.5, suffix_cap=cap)
    rng = np.random.default_rng(docs)
    gen = torch.Generator(device="cuda").manual_seed(docs)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=gen).to(torch.bfloat16)                 # noqa: E731
    q, pk, pv, sk, sv = rnd(n, Hq, D), rnd(T, Hkv, D), rnd(T, Hkv, D), rnd(n * cap, Hkv, D), rnd(n * cap, Hkv, D)
    depth, alive = dev(rng.integers(0, cap, n).astype(np.int32)), dev(np.ones(n, np.uint8))
    vis = dev(rng.integers(0, np.repeat(L, cnt) + 1).astype(np.int32))
    m = B.MetaTables.alloc(g, docs + 1, n, T)
    if order:
        B.hpd_build_meta_skeleton(g, docs + 1, n, dev(L), dev(cnt), depth, alive, vis, 0, m)
    else:
        B.hpd_build_meta(g, docs + 1, n, dev(L), dev(cnt), depth, alive, 0, m)

    def attn(m, q, rows):
        o, lse = torch.zeros(rows, Hq, D, dtype=torch.bfloat16, device="cuda"), torch.zeros(rows, Hq, device="cuda")
        if order:
            B.hpd_attn_decode_posorder(g, docs + 1, rows, n, T, q, pk, pv, sk, sv, dev(L), depth, alive, m, True, o, lse)
        else:
            B.hpd_attn_decode(g, docs + 1, rows, n, T, q, pk, pv, sk, sv, dev(L), m, True, o, lse)
        torch.cuda.synchronize()
        return o, lse

    def later(t, fill):
        return torch.cat([torch.full((MOVED,), fill, dtype=t.dtype, device="cuda"), t])
    want, want_lse = attn(m, q, n)
    moved = replace(m, doc_active_start=m.doc_active_start + MOVED, n_active=m.n_active + MOVED, doc_id=later(m.doc_id, docs),
                    **{k: later(getattr(m, k), 0) for k in ("active_slot", "suffix_off", "suffix_len", "prefix_vis")})
    got, got_lse = attn(moved, torch.cat([rnd(MOVED, Hq, D), q]), n + MOVED)
    assert int(m.dev_status.item()) == 0
    assert torch.equal(got[MOVED:], want) and torch.equal(got_lse[MOVED:], want_lse)
    assert not got[:MOVED].any() and not got_lse[:MOVED].any()
