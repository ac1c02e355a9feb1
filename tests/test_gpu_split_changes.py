"""Steps that split documents and steps that do not, in turn on one workspace and without waiting in between: the merge kernel looks at the
plan before its predecessor has ended, and most of its blocks end there when nothing was split."""
import pytest
import torch

from paper_2604_26209_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("docs,live_docs", [(64, 1), (40, 3), (12, 1)])
def test_split_and_whole_steps_alternate(docs, live_docs, captured):
    from paper_2604_26209_b200 import binding as B
    g = synth.Geom(Hq=32, Hkv=8, D=128, rope_theta=500000.0, sm_scale=128 ** -0.5, suffix_cap=4)
    branches, L = 3, 1600                                             # a lone document: four chunks of 512
    n, T = docs * branches, docs * L
    rows = live_docs * branches
    gen = torch.Generator(device="cuda").manual_seed(docs)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=gen).to(torch.bfloat16)                                   # noqa: E731
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")                                                   # noqa: E731
    pk, pv, sk, sv, q = rnd(T, 8, 128), rnd(T, 8, 128), rnd(n * 4, 8, 128), rnd(n * 4, 8, 128), rnd(n, 32, 128)
    lens, cnt, depth = i32([L] * docs), i32([branches] * docs), i32([s % 4 for s in range(n)])
    every = torch.ones(n, dtype=torch.uint8, device="cuda")
    few = torch.zeros(n, dtype=torch.uint8, device="cuda")
    few[-rows:] = 1
    q[-rows:] = q[:rows]                                              # the live rows of both kinds of step are the same
    m = B.MetaTables.alloc(g, docs, n, T)

    def steps(outs, wait):
        for i, o in enumerate(outs):
            B.hpd_build_meta(g, docs, n, lens, cnt, depth, few if i % 2 else every, 0, m)
            for _ in range(2):                                        # two layers: the ticket counter is rewound in between
                B.hpd_attn_decode(g, docs, n, n, T, q, pk, pv, sk, sv, lens, m, False, o[0], o[1])
                if wait:
                    torch.cuda.synchronize()

    new = lambda: [(torch.zeros(n, 32, 128, dtype=torch.bfloat16, device="cuda"), torch.zeros(n, 32, device="cuda")) for _ in range(6)]  # noqa: E731
    want, got = new(), new()
    steps(want, True)
    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            steps(got, False)
        graph.replay()
        graph.replay()
    else:
        steps(got, False)
    torch.cuda.synchronize()
    assert int(m.dev_status.item()) == 0
    for (o, lse), (o2, lse2) in zip(want, got):
        assert torch.equal(o, o2) and torch.equal(lse, lse2)
    # a split step's rows are the whole step's rows: same keys, other order of summation (bf16 outputs, fp32 partials)
    assert (want[1][0][:rows].float() - want[0][0][-rows:].float()).abs().max().item() <= 2e-2
    assert (want[1][1][:rows] - want[0][1][-rows:]).abs().max().item() <= 1e-3
