"""What users of this framework run on the GPU, as cases that can be timed: the decode step over stacked documents, the
same step under the position-order mask and with a block shared by all documents, the first inference step, and the decode
loop with retirement.  Every case goes through the Python binding of the C ABI, one call per operation, as a model's
attention layers call it.

    listed()            the cases by name
    draw(rng)           one more case of the same ranges
    prepare(case, seed) a user's state: caches, activations, slot tables, table and workspace memory
    run(state)          one pass: tables, rotary embedding + append, attention (and the end of the step in the loop)
    work(case)          bytes and operations a pass cannot do without
    tolerance(case)     what another correct implementation at the same precision may differ by

A case is a dict of plain values.  `kind` names the path:
    decode    prompts x docs documents of len_lo..len_hi prefix tokens, `branches` branches each, depth 0..depth_hi-1 of a slab of
              `cap`, a share `alive` of them still decoding, position gap 0 or cap; mask: own document, own branch
    posorder  prompts groups of len_lo..len_hi prompt tokens + 1..4 skeleton tokens per branch; mask: position order
    shared    decode with `block` tokens in front of every document, stored once
    prefill   the first inference step of the posorder structure: every prompt token is a row
    loop      the decode structure from depth 0 for cap steps; a value ends after each token with probability 1/mean; one step (tables,
              all layers, end of step) is a CUDA graph that is replayed, as a server that does not want a host call per kernel does
"""
import numpy as np
import torch

from paper_2604_26209_b200 import binding as B
from paper_2604_26209_b200.synth import Geom

KEY_HI = 4                                   # skeleton: attribute keys of 1..4 tokens
LLAMA = dict(Hq=32, Hkv=8, D=128)            # the benchmark's attention geometry (Llama-3-8B)
MAIN = dict(docs=4, len_lo=512, len_hi=512, branches=24, cap=16, depth_hi=16, alive=1.0, gap=0, layers=1, lse=True, **LLAMA)
STACKED = dict(len_lo=2048, len_hi=2048, branches=96, cap=16, depth_hi=16, alive=1.0, layers=1, **LLAMA)


def listed():
    return [
        # one short document, four attributes, a small head geometry: nothing but latency and launches
        dict(name="decode_tiny", kind="decode", prompts=1, docs=1, len_lo=256, len_hi=256, branches=4, cap=8, depth_hi=8, alive=1.0,
             gap=0, layers=1, lse=True, Hq=4, Hkv=1, D=64),
        # one product page answered interactively: 96 branches
        dict(MAIN, name="decode_1_prompt", kind="decode", prompts=1),
        # a small batch, its caches still in L2
        dict(MAIN, name="decode_8_prompts", kind="decode", prompts=8),
        # the benchmark's own workload: a full batch of stacked documents
        dict(MAIN, name="decode_64_prompts", kind="decode", prompts=64),
        # long documents of ragged length, few branches each
        dict(MAIN, name="decode_long", kind="decode", prompts=32, docs=8, len_lo=1024, len_hi=4096, branches=12, cap=32, depth_hi=32),
        # the paper's own prompt (6 documents x 16 attributes, K_max = 30) some way into decoding: odd lengths, half the branches retired,
        # Algorithm 2's position gaps, 8 query heads per kv head, two layers
        dict(name="decode_paper_shape", kind="decode", prompts=11, docs=6, len_lo=83, len_hi=1277, branches=16, cap=30, depth_hi=30,
             alive=0.5, gap=30, layers=2, lse=False, Hq=32, Hkv=4, D=128),
        # the mask the paper's implementation runs, for one prompt and for a full batch
        dict(STACKED, name="posorder_1_prompt", kind="posorder", prompts=1, lse=False),
        dict(STACKED, name="posorder_64_prompts", kind="posorder", prompts=64, lse=True),
        # instruction and attribute definitions stored once in front of all documents
        dict(MAIN, name="shared_64_prompts", kind="shared", prompts=64, len_lo=384, len_hi=384, block=128),
        # the first inference step (prefill) of one prompt and of a full batch
        dict(STACKED, name="prefill_1_prompt", kind="prefill", prompts=1, lse=False),
        dict(STACKED, name="prefill_64_prompts", kind="prefill", prompts=64, lse=False),
        # a whole batch decoded to its end: four layers, branches retiring, one graph per step
        dict(MAIN, name="loop_16_prompts", kind="loop", prompts=16, cap=32, layers=4, mean=8, lse=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "decode", "posorder", "posorder", "shared", "prefill", "prefill", "loop"])
    Hq, Hkv, D = rng.choice([(32, 8, 128)] * 4 + [(32, 4, 128), (16, 8, 128), (8, 8, 128), (4, 1, 64), (8, 4, 64), (8, 1, 64)])
    lo = _log_int(rng, 16, 3000)
    c = dict(kind=kind, prompts=_log_int(rng, 1, 64), len_lo=lo, len_hi=min(4096, lo + int(lo * rng.choice([0, 0.3, 1, 3]))),
             branches=_log_int(rng, 1, 48), cap=rng.choice([5, 8, 16, 16, 30, 32]), alive=rng.choice([1.0, 1.0, 0.7, 0.3]),
             layers=rng.choice([1, 1, 2, 4]), lse=rng.random() < 0.5, Hq=Hq, Hkv=Hkv, D=D)
    c["depth_hi"] = rng.randint(1, c["cap"])
    if kind in ("posorder", "prefill"):
        c["branches"] = _log_int(rng, 4, 128)
    else:
        c["docs"] = rng.randint(1, 8)
        c["gap"] = rng.choice([0, c["cap"]])
    if kind == "shared":
        c["gap"], c["block"] = 0, _log_int(rng, 16, 600)
    if kind == "loop":
        c.update(alive=1.0, depth_hi=1, mean=rng.choice([4, 8, 12]), layers=rng.choice([1, 2, 4]))
    # no drawn case costs more than the listed ones: fewer prompts, then fewer layers, until it does not
    big = {"prefill": (9e9, 2.6e12), "loop": (25e9, 2e12)}.get(kind, (2.9e9, 0.26e12))
    while c["prompts"] > 1 or c["layers"] > 1:
        w = work(c)
        if w["bytes"] <= big[0] and w["flops"] <= big[1]:
            break
        if c["prompts"] > 1:
            c["prompts"] = max(1, c["prompts"] * 3 // 4)
        else:
            c["layers"] -= 1
    return c


# ---------------------------------------------------------------------------------------------------------------------
def _structure(c, rng):
    """Document lengths, slots per document, depths, live flags, and per slot the prefix tokens it sees (skeleton).  Lengths belong
    to the case, their order to the seed: a case's totals are the same for every seed."""
    own = np.random.default_rng([c["prompts"], c["len_lo"], c["len_hi"], c["branches"]])
    groups = c["kind"] in ("posorder", "prefill")
    n_docs = c["prompts"] * (1 if groups else c["docs"])
    L = rng.permutation(own.integers(c["len_lo"], c["len_hi"] + 1, size=n_docs, dtype=np.int32))
    cnt = np.full(n_docs, c["branches"], np.int32)
    n = int(cnt.sum())
    vis = None
    if groups:
        key = rng.permutation(own.integers(1, KEY_HI + 1, size=n_docs * c["branches"])).reshape(n_docs, -1).cumsum(axis=1)
        vis = (L[:, None] + key).astype(np.int32).reshape(-1)
        L = (L + key[:, -1]).astype(np.int32)
    if c["kind"] == "shared":
        vis = np.repeat(L + c["block"], c["branches"]).astype(np.int32)
    depth = rng.integers(0, c["depth_hi"], size=n, dtype=np.int32)
    alive = (rng.random(n) < c["alive"]).astype(np.uint8)
    alive[0] = 1
    return L, cnt, depth, alive, vis


def prepare(case, seed):
    c = case
    rng = np.random.default_rng([seed & 0x7FFFFFFF, 0x485044])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed & 0x7FFFFFFFFFFF)
    L, cnt, depth, alive, vis = _structure(c, rng)
    g = Geom(Hq=c["Hq"], Hkv=c["Hkv"], D=c["D"], rope_theta=500000.0, sm_scale=float(c["D"]) ** -0.5, suffix_cap=c["cap"])
    n_docs, n, T = len(L), len(depth), int(L.sum())
    gpu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()                                                    # noqa: E731
    rnd = lambda *shape: torch.randn(*shape, device="cuda", dtype=torch.bfloat16, generator=gen)                        # noqa: E731
    s = dict(c=c, g=g, n_docs=n_docs, n=n, T=T, L=gpu(L), cnt=gpu(cnt), depth=gpu(depth), alive=gpu(alive),
             vis=None if vis is None else gpu(vis))
    if c["kind"] == "prefill":
        # the layers' projections have been written: queries and outputs per layer, keys and values in the prefix cache
        s["layers"] = [dict(q=rnd(T, g.Hq, g.D), pk=rnd(T, g.Hkv, g.D), pv=rnd(T, g.Hkv, g.D),
                            o=torch.zeros(T, g.Hq, g.D, dtype=torch.bfloat16, device="cuda"),
                            lse=torch.zeros(T, g.Hq, device="cuda") if c["lse"] else None) for _ in range(c["layers"])]
        s["t"] = B.PrefillTables.alloc(g, n_docs, T)
        return s
    rows = n * g.suffix_cap
    s["layers"] = [dict(q=rnd(n, g.Hq, g.D), k=rnd(n, g.Hkv, g.D), v=rnd(n, g.Hkv, g.D), pk=rnd(T, g.Hkv, g.D), pv=rnd(T, g.Hkv, g.D),
                        sk=rnd(rows, g.Hkv, g.D), sv=rnd(rows, g.Hkv, g.D),
                        o=torch.zeros(n, g.Hq, g.D, dtype=torch.bfloat16, device="cuda"),
                        lse=torch.zeros(n, g.Hq, device="cuda") if c["lse"] else None) for _ in range(c["layers"])]
    s["m"] = B.MetaTables.alloc(g, n_docs, n, T)
    if c["kind"] == "shared":
        for y in s["layers"]:
            y.update(bk=rnd(c["block"], g.Hkv, g.D), bv=rnd(c["block"], g.Hkv, g.D))
        s.update(doc_block=torch.zeros(n_docs, dtype=torch.int32, device="cuda"), block_start=gpu(np.zeros(1, np.int32)),
                 block_len=gpu(np.full(1, c["block"], np.int32)))
    if c["kind"] == "loop":
        # sampled tokens of every step (0 is the delimiter), the step as a graph
        s["tokens"] = torch.randint(0, c["mean"], (c["cap"], n), dtype=torch.int32, device="cuda", generator=gen)
        s["token"] = torch.ones(n, dtype=torch.int32, device="cuda")
        s["n_alive"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        _loop_reset(s)
        _loop_step(s)                        # the first call sets kernel attributes
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _loop_step(s)
    return s


# ---------------------------------------------------------------------------------------------------------------------
def _rope_append(s, y):
    m = s["m"]
    B.hpd_rope_append(s["g"], s["n"], s["n"], m.n_active, m.pos_id, m.suffix_off, m.suffix_len, y["q"], y["k"], y["v"], y["sk"], y["sv"],
                      m.dev_status)


def _attn(s, y):
    B.hpd_attn_decode(s["g"], s["n_docs"], s["n"], s["n"], s["T"], y["q"], y["pk"], y["pv"], y["sk"], y["sv"], s["L"], s["m"], True,
                      y["o"], y["lse"])


def _loop_reset(s):
    s["depth"].zero_()
    s["alive"].fill_(1)


def _loop_step(s):
    m, g = s["m"], s["g"]
    B.hpd_build_meta(g, s["n_docs"], s["n"], s["L"], s["cnt"], s["depth"], s["alive"], s["c"]["gap"], m)
    for y in s["layers"]:
        _rope_append(s, y)
        _attn(s, y)
    B.hpd_advance(g, s["n"], m.n_active, m.active_slot, s["token"], 0, s["depth"], s["alive"], s["n_alive"])


def _tables(m):
    names = m.NAMES + ("n_active", "dev_status")
    return {k: getattr(m, k) for k in names}


def run(state):
    s = state
    c, g = s["c"], s["g"]
    if c["kind"] == "prefill":
        t = s["t"]
        B.hpd_prefill_meta(g, s["n_docs"], s["n"], s["T"], s["L"], s["cnt"], s["vis"], c["cap"], t)
        for y in s["layers"]:
            B.hpd_rope(g, s["T"], t.n_tokens, t.tok_pos, y["q"], y["pk"])
            B.hpd_prefill_attn(g, s["n_docs"], s["T"], y["q"], y["pk"], y["pv"], s["L"], t, y["o"], y["lse"])
        return {"layers": [{k: y[k] for k in ("o", "lse", "q", "pk")} for y in s["layers"]],
                "tables": [t.doc_kv_start, t.doc_slot_start, t.tok_doc, t.tok_pos, t.tok_vis, t.n_tokens, t.dev_status]}
    m = s["m"]
    if c["kind"] == "loop":
        _loop_reset(s)
        for step in range(c["cap"]):
            s["token"].copy_(s["tokens"][step])
            s["graph"].replay()
        return {"layers": [{k: y[k] for k in ("o", "q", "k", "sk", "sv")} for y in s["layers"]], "tables": _tables(m),
                "depth": s["depth"], "alive": s["alive"], "n_alive": s["n_alive"]}
    if c["kind"] == "decode":
        B.hpd_build_meta(g, s["n_docs"], s["n"], s["L"], s["cnt"], s["depth"], s["alive"], c["gap"], m)
    else:
        B.hpd_build_meta_skeleton(g, s["n_docs"], s["n"], s["L"], s["cnt"], s["depth"], s["alive"], s["vis"],
                                  c["cap"] if c["kind"] == "posorder" else 0, m)
    for y in s["layers"]:
        _rope_append(s, y)
        if c["kind"] == "decode":
            _attn(s, y)
        elif c["kind"] == "posorder":
            B.hpd_attn_decode_posorder(g, s["n_docs"], s["n"], s["n"], s["T"], y["q"], y["pk"], y["pv"], y["sk"], y["sv"], s["L"],
                                       s["depth"], s["alive"], m, True, y["o"], y["lse"])
        else:
            B.hpd_attn_decode_shared(g, s["n_docs"], s["n"], s["n"], s["T"], y["q"], y["pk"], y["pv"], y["sk"], y["sv"], y["bk"], y["bv"],
                                     c["block"], s["doc_block"], s["block_start"], s["block_len"], s["L"], m, True, y["o"], y["lse"])
    return {"layers": [{k: y[k] for k in ("o", "lse", "q", "k", "sk", "sv")} for y in s["layers"]], "tables": _tables(m)}


# ---------------------------------------------------------------------------------------------------------------------
def work(case):
    """Expected bytes and operations of a pass (lengths and depths are drawn per seed: their means)."""
    c = case
    Hq, Hkv, D = c["Hq"], c["Hkv"], c["D"]
    kv, head = 2 * Hkv * D * 2, Hq * D * 2                       # K + V of one token; one row's q or o
    Lm = (c["len_lo"] + c["len_hi"]) / 2
    var = (c["len_hi"] - c["len_lo"]) ** 2 / 12
    lse = Hq * 4 if c["lse"] else 0
    if c["kind"] in ("posorder", "prefill"):
        skel = c["branches"] * (1 + KEY_HI) / 2
        Lp, groups = Lm + skel, c["prompts"]
        if c["kind"] == "prefill":
            T = groups * Lp
            pairs = groups * ((Lp * Lp + var) + Lp) / 2
            return {"bytes": c["layers"] * T * (3 * head + 1.5 * kv + lse) + 12 * T, "flops": c["layers"] * 4 * D * Hq * pairs}
        rows = groups * c["branches"] * c["alive"]
        cached = groups * c["branches"] * (c["depth_hi"] - 1) / 2          # retired branches' tokens stay visible
        keys = rows * (Lm + skel / 2 + ((c["depth_hi"] - 1) / 2 + c["alive"]) * c["branches"] / 2)
        return {"bytes": c["layers"] * (groups * Lp * kv + cached * kv + rows * (3 * head + 2.5 * kv + lse)) + 28 * groups * c["branches"],
                "flops": c["layers"] * 4 * D * Hq * keys}
    docs = c["prompts"] * c["docs"]
    slots = docs * c["branches"]
    blk = c.get("block", 0)

    def step(p_alive, depth):
        rows = slots * p_alive
        live = docs * (1 - (1 - p_alive) ** c["branches"])
        return (c["layers"] * (live * Lm * kv + blk * kv + rows * depth * kv + rows * (3 * head + 2.5 * kv + lse)) + 28 * slots,
                c["layers"] * 4 * D * Hq * rows * (Lm + blk + depth + 1))

    if c["kind"] == "loop":
        parts = [step((1 - 1 / c["mean"]) ** t, t) for t in range(c["cap"])]
    else:
        parts = [step(c["alive"], (c["depth_hi"] - 1) / 2)]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    # bf16 outputs of sums over bf16 probabilities: 2.3e-3 (2-norm) and 1.4e-2 (largest) away from the same step in 64 bits; four
    # times that.  Tables, depths and flags are whole numbers and exact.
    return {"rel": 9e-3, "max": 0.055, "differ": 0.0}
