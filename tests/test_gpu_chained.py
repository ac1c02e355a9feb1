"""Order between chained calls and everything around them.  A kernel may be resident while its predecessor in the stream still writes:
nothing it reads may be older than that, whatever stands in front of it."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import synth
from tests.util import err_stats, oracle_step

pytestmark = pytest.mark.gpu

LAYERS = 2
# documents, branches, slab, prefix lengths, (Hq, Hkv, D): a few blocks; a wave of CTAs; one split document (the merge has work); more
# than 8192 rows (the end of the step is a memset and many blocks)
SHAPES = {"small": (3, 5, 4, (40, 200), (2, 1, 64)), "wave": (32, 24, 6, (300, 600), (8, 2, 128)), "split": (1, 4, 4, (3000, 3000), (8, 2, 128)),
          "rows": (411, 20, 3, (8, 40), (2, 1, 64))}


def _loop_state(shape):
    docs, branches, cap, (lo, hi), (Hq, Hkv, D) = SHAPES[shape]
    g = synth.Geom(Hq=Hq, Hkv=Hkv, D=D, rope_theta=10000.0, sm_scale=D ** -0.5, suffix_cap=cap)
    rng = np.random.default_rng(docs)
    gen = torch.Generator(device="cuda").manual_seed(docs)
    n, steps = docs * branches, cap + 1
    L = rng.integers(lo, hi + 1, docs).astype(np.int32)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=gen).to(torch.bfloat16)                 # noqa: E731
    c = dict(L=torch.from_numpy(L).cuda(), cnt=torch.full((docs,), branches, dtype=torch.int32, device="cuda"),
             pk=[rnd(int(L.sum()), Hkv, D) for _ in range(LAYERS)], pv=[rnd(int(L.sum()), Hkv, D) for _ in range(LAYERS)],
             token=torch.from_numpy(rng.integers(0, 4, (steps, n)).astype(np.int32)).cuda())          # 0 ends the value
    s = dict(depth=torch.zeros(n, dtype=torch.int32, device="cuda"), alive=torch.ones(n, dtype=torch.uint8, device="cuda"),
             n_alive=torch.zeros(steps, dtype=torch.int32, device="cuda"))
    for l in range(LAYERS):
        s[f"sk{l}"], s[f"sv{l}"] = rnd(n * cap, Hkv, D), rnd(n * cap, Hkv, D)
        for t in range(steps):
            s[f"q{t}{l}"], s[f"k{t}{l}"], s[f"v{t}{l}"] = rnd(n, Hq, D), rnd(n, Hkv, D), rnd(n, Hkv, D)
            s[f"o{t}{l}"], s[f"lse{t}{l}"] = torch.zeros(n, Hq, D, dtype=torch.bfloat16, device="cuda"), torch.zeros(n, Hq, device="cuda")
    return g, docs, n, steps, int(L.sum()), c, s


@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_back_to_back_steps_equal_synchronised_ones(shape):
    """Several steps of two layers with nothing between the calls, direct and as one graph, bit for bit as with a wait after each."""
    from paper_2604_26209_b200 import binding as B
    g, docs, n, steps, T, c, s = _loop_state(shape)
    start = {k: v.clone() for k, v in s.items()}
    m = B.MetaTables.alloc(g, docs, n, T)
    m.workspace.zero_()

    def run(wait):
        def call(f, *a):
            f(*a)
            if wait:
                torch.cuda.synchronize()
        for t in range(steps):
            call(B.hpd_build_meta, g, docs, n, c["L"], c["cnt"], s["depth"], s["alive"], 0, m)
            for l in range(LAYERS):
                call(B.hpd_rope_append, g, n, n, m.n_active, m.pos_id, m.suffix_off, m.suffix_len, s[f"q{t}{l}"], s[f"k{t}{l}"], s[f"v{t}{l}"],
                     s[f"sk{l}"], s[f"sv{l}"], m.dev_status)
                call(B.hpd_attn_decode, g, docs, n, n, T, s[f"q{t}{l}"], c["pk"][l], c["pv"][l], s[f"sk{l}"], s[f"sv{l}"], c["L"], m, True,
                     s[f"o{t}{l}"], s[f"lse{t}{l}"])
            call(B.hpd_advance, g, n, m.n_active, m.active_slot, c["token"][t], 0, s["depth"], s["alive"], s["n_alive"][t:t + 1])

    def result(f):
        for k, v in start.items():
            s[k].copy_(v)
        for name in m.NAMES + ("n_active",):             # tables that would be followed if they were read too early, all in range
            getattr(m, name).zero_()
        torch.cuda.synchronize()
        f()
        torch.cuda.synchronize()
        assert int(m.dev_status.item()) == 0
        out = dict(s, **{name: getattr(m, name) for name in m.NAMES + ("n_active",)})
        return {k: v.clone().view(torch.int16) if v.dtype == torch.bfloat16 else v.clone().view(torch.int32) if v.is_floating_point() else v.clone()
                for k, v in out.items()}

    want = result(lambda: run(True))
    counts = want["n_alive"].tolist()
    assert counts[-1] == 0 and all(a >= b for a, b in zip(counts, counts[1:]))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run(False)
    for f in (lambda: run(False), graph.replay, lambda: run(False), graph.replay):
        got = result(f)
        for k in want:
            assert torch.equal(got[k], want[k]), k


@pytest.mark.parametrize("direct", [True, False])
def test_calls_behind_events_copies_and_ordinary_kernels(direct):
    """Two steps with other inputs and other live branches, copied in by a second stream and out by a third, without a host wait; the
    calls stand behind the event (direct) or behind ordinary kernels that write their inputs.  Against the oracle."""
    from paper_2604_26209_b200 import runtime
    base = synth.config_custom("edges", Hq=8, Hkv=2, D=128, theta=10000.0, cap=6, prefix_lens=[(97 * i) % 700 for i in range(24)], branch_cnts=[8] * 24,
                               depth_hi=6, seed=11, alive_frac=0.8)
    rng = np.random.default_rng(12)
    structs = [base, replace(base, slot_depth=rng.integers(0, 6, base.n_slots).astype(np.int32),
                             slot_alive=(rng.random(base.n_slots) < 0.4).astype(np.uint8))]
    tbs = [synth.make_tensors(base), synth.make_tensors(base, salt=5)]
    wants = [oracle_step(s, tb) for s, tb in zip(structs, tbs)]
    db = runtime.DeviceBatch(base, dict(tbs[0], suffix_k=np.zeros_like(tbs[0]["suffix_k"]), suffix_v=np.zeros_like(tbs[0]["suffix_v"])))
    bits = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).view(torch.bfloat16)    # noqa: E731
    targets = dict(depth=db.slot_depth, alive=db.slot_alive, q=db.q, k=db.k_new, v=db.v_new, sk=db.suffix_k, sv=db.suffix_v, pk=db.prefix_k,
                   pv=db.prefix_v)
    hosts, stages, outs = [], [], []
    for s, tb, (meta, _) in zip(structs, tbs, wants):
        act = np.concatenate([meta.active_slot[:meta.n_active], np.setdiff1d(np.arange(s.n_slots), meta.active_slot[:meta.n_active])])
        h = dict(depth=torch.from_numpy(s.slot_depth), alive=torch.from_numpy(s.slot_alive), q=bits(tb["q"][act]), k=bits(tb["k_new"][act]),
                 v=bits(tb["v_new"][act]), sk=bits(tb["suffix_k"]), sv=bits(tb["suffix_v"]), pk=bits(tb["prefix_k"]), pv=bits(tb["prefix_v"]))
        hosts.append({k: v.reshape(targets[k].shape).pin_memory() for k, v in h.items()})
        stages.append({k: torch.empty_like(v) for k, v in targets.items()})
        outs.append(dict(o=torch.empty(db.o.shape, dtype=db.o.dtype).pin_memory(), lse=torch.empty(db.lse.shape).pin_memory()))
    db.step()                                            # kernel attributes, tensor maps
    ballast = torch.zeros(2, 1 << 25, device="cuda")
    compute, copy_in, copy_out = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    free = None
    for h, stage, out in zip(hosts, stages, outs):
        with torch.cuda.stream(copy_in):
            if free is not None:                         # the step before has been read
                copy_in.wait_event(free)
            ballast[1].copy_(ballast[0])                 # the inputs come late
            for k in h:
                (targets[k] if direct else stage[k]).copy_(h[k], non_blocking=True)
            ready = copy_in.record_event()
        with torch.cuda.stream(compute):
            compute.wait_event(ready)
            if not direct:
                for k in ("depth", "alive", "sk", "sv", "pk", "pv"):
                    targets[k].copy_(stage[k])
            db.build_meta()
            if not direct:
                for k in ("q", "k", "v"):
                    targets[k].copy_(stage[k])
            db.rope_append()
            db.attn(True)
            done = compute.record_event()
        with torch.cuda.stream(copy_out):
            copy_out.wait_event(done)
            out["o"].copy_(db.o, non_blocking=True)
            out["lse"].copy_(db.lse, non_blocking=True)
            free = copy_out.record_event()
    torch.cuda.synchronize()
    assert db.status() == 0
    assert wants[0][0].n_active != wants[1][0].n_active
    for out, (meta, want) in zip(outs, wants):
        n = meta.n_active
        mx, mean = err_stats(out["o"][:n].float().numpy(), want.o)
        assert mx <= 2e-2 and mean <= 2e-3, (mx, mean)
        assert np.max(np.abs(out["lse"][:n].numpy() - want.lse)) <= 2e-2


@pytest.mark.parametrize("side", ["copy", "kernel"])
def test_captured_calls_behind_a_join_of_two_streams(side):
    """A graph in which each call also depends on another stream's copy or kernel that writes its inputs, against the step without them."""
    from paper_2604_26209_b200 import runtime
    s = synth.config_custom("join", Hq=8, Hkv=2, D=128, theta=10000.0, cap=6, prefix_lens=[300] * 16, branch_cnts=[8] * 16, depth_hi=5, seed=21,
                            alive_frac=0.7)
    tb = synth.make_tensors(s)
    meta, want = oracle_step(s, tb)
    act = np.concatenate([meta.active_slot[:meta.n_active], np.setdiff1d(np.arange(s.n_slots), meta.active_slot[:meta.n_active])])
    db = runtime.DeviceBatch(s, tb)
    inputs = [(db.q, tb["q"][act]), (db.k_new, tb["k_new"][act]), (db.v_new, tb["v_new"][act])]
    inputs = [(t, torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda().view(torch.bfloat16).reshape(t.shape)) for t, a in inputs]
    tables = [(db.slot_depth, db.slot_depth.clone()), (db.slot_alive, db.slot_alive.clone())]
    write = (lambda t, a: t.copy_(a)) if side == "copy" else (lambda t, a: torch.mul(a, 1, out=t))    # a memcpy node, a kernel node
    db.step()
    other = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()

    def beside(pairs):
        main = torch.cuda.current_stream()
        other.wait_stream(main)
        with torch.cuda.stream(other):
            for t, a in pairs:
                write(t, a)
        return lambda: main.wait_stream(other)

    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        beside(tables)()
        join = beside(inputs)
        db.build_meta()
        join()
        db.rope_append()
        join = beside([(db.lse, torch.zeros_like(db.lse))])
        join()
        db.attn(True)
    for _ in range(3):
        db.q.zero_(); db.k_new.zero_(); db.v_new.zero_(); db.o.zero_(); db.slot_alive.zero_(); db.slot_depth.fill_(1)
        graph.replay()
        torch.cuda.synchronize()
        assert db.status() == 0 and int(db.meta.n_active.item()) == meta.n_active
        mx, mean = err_stats(synth.bf16_bits_to_f32(runtime.bits_of(db.o))[:meta.n_active], want.o)
        assert mx <= 2e-2 and mean <= 2e-3, (mx, mean)
        assert np.max(np.abs(db.lse.cpu().numpy()[:meta.n_active] - want.lse)) <= 2e-2


@pytest.mark.parametrize("tokens", [40, 900, 5000])      # a few CTAs, about one wave of the rotation, more than one
def test_back_to_back_first_steps_equal_synchronised_ones(tokens):
    """Two first inference steps of two layers, with nothing between the calls, bit for bit as with a wait after each."""
    from paper_2604_26209_b200 import binding as B
    g = synth.Geom(Hq=8, Hkv=2, D=128, rope_theta=10000.0, sm_scale=128 ** -0.5, suffix_cap=8)
    L = torch.tensor([tokens // 3, tokens - tokens // 3], dtype=torch.int32, device="cuda")
    vis = torch.tensor([tokens // 6, tokens // 3, tokens // 5, tokens // 2], dtype=torch.int32, device="cuda")
    cnt = torch.tensor([2, 2], dtype=torch.int32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(tokens)
    start = [torch.randn(tokens, h, 128, device="cuda", generator=gen).to(torch.bfloat16) for _ in range(2 * LAYERS) for h in (8, 2, 2)]
    t = B.PrefillTables.alloc(g, 2, tokens)

    def run(wait):
        for x in (t.doc_kv_start, t.doc_slot_start, t.tok_doc, t.tok_pos, t.tok_vis, t.n_tokens, t.workspace):
            x.zero_()
        work = [x.clone() for x in start]
        outs = [torch.zeros_like(start[0]) for _ in range(2 * LAYERS)]
        sync = torch.cuda.synchronize if wait else (lambda: None)
        torch.cuda.synchronize()
        for step in range(2):
            B.hpd_prefill_meta(g, 2, 4, tokens, L, cnt, vis, 8, t); sync()
            for l in range(step * LAYERS, (step + 1) * LAYERS):
                q, k, v = work[3 * l:3 * l + 3]
                B.hpd_rope(g, tokens, t.n_tokens, t.tok_pos, q, k); sync()
                B.hpd_prefill_attn(g, 2, tokens, q, k, v, L, t, outs[l]); sync()
        torch.cuda.synchronize()
        assert int(t.dev_status.item()) == 0
        return [x.view(torch.int16) for x in work + outs] + [x.clone() for x in (t.tok_doc, t.tok_pos, t.tok_vis, t.n_tokens)]

    want = run(True)
    for _ in range(3):
        assert all(torch.equal(a, b) for a, b in zip(run(False), want))
