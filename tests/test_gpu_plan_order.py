"""The work list of steps whose documents differ in length: longest unit first, every document once, at the list sizes where the plan's
ordering changes its method (counting up to 512 keys, a sorting network of up to 2048 beyond) or pads its keys."""
import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("docs", [2, 63, 64, 65, 127, 129, 256, 257, 511, 512, 513, 1024, 1025, 2048])
def test_list_is_longest_first(docs):
    from paper_2604_26209_b200 import binding as B
    rng = np.random.default_rng(docs)
    L = rng.integers(1, 400, size=docs).astype(np.int32)              # ties among them: document order decides
    L[0], L[-1] = 500, 1                                              # below a chunk (512): documents stay whole
    dev = lambda a: torch.from_numpy(a).cuda()                        # noqa: E731
    g = synth.Geom(Hq=2, Hkv=1, D=64, rope_theta=10000.0, sm_scale=0.125, suffix_cap=4)
    m = B.MetaTables.alloc(g, docs, docs, int(L.sum()))
    B.hpd_build_meta(g, docs, docs, dev(L), dev(np.ones(docs, np.int32)), dev(np.zeros(docs, np.int32)), dev(np.ones(docs, np.uint8)), 0, m)
    torch.cuda.synchronize()
    words = m.workspace.cpu().numpy().view(np.uint8)[: 256 + 32 * docs].view(np.int32)
    items = words[64:].reshape(docs, 8)                               # document, first key, keys, ... behind the 256-byte header
    assert words[0] == docs
    assert np.array_equal(items[:, 2], L[items[:, 0]]) and not items[:, 1].any()
    # equal costs (branches are equal, so equal lengths) keep document order
    assert np.array_equal(items[:, 0], np.lexsort((np.arange(docs), -L.astype(np.int64))))
