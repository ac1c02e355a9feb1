"""An error that one call reports is not reported again by the next."""
import ctypes as C

import pytest
import torch

from paper_2604_26209_b200 import synth

pytestmark = pytest.mark.gpu


def test_failed_launch_leaves_no_error_for_the_next_call():
    from paper_2604_26209_b200 import binding as B
    g = synth.Geom(Hq=2, Hkv=1, D=64, rope_theta=10000.0, sm_scale=0.125, suffix_cap=4)
    i32 = lambda v: torch.tensor([v], dtype=torch.int32, device="cuda")                     # noqa: E731
    q, k, sk, sv = (torch.ones(n, h, 64, dtype=torch.bfloat16, device="cuda") for n, h in ((1, 2), (1, 1), (4, 1), (4, 1)))
    n, zero, status = i32(1), i32(0), i32(0)
    v = 3 * k
    torch.cuda.synchronize()
    # a capture that an illegal call has ended: launches into the stream are refused by the runtime
    rt, s = C.CDLL("libcudart.so.12"), torch.cuda.Stream()
    handle, graph = C.c_void_p(s.cuda_stream), C.c_void_p()
    assert rt.cudaStreamBeginCapture(handle, 2) == 0
    try:
        assert rt.cudaStreamSynchronize(handle) != 0
        with torch.cuda.stream(s), pytest.raises(B.HpdError):
            B.hpd_rope(g, 1, n, zero, q, k)
    finally:
        rt.cudaStreamEndCapture(handle, C.byref(graph))
        rt.cudaGetLastError()
    B.hpd_kv_append(g, 1, 1, n, zero, zero, k, v, sk, sv, status)
    torch.cuda.synchronize()
    assert torch.equal(sk[0], k[0]) and torch.equal(sv[0], v[0]) and int(status.item()) == 0


def test_every_native_call_refuses_tensors_with_other_strides():
    """A pointer says nothing of strides: each call refuses a tensor that is not dense, whichever argument it is."""
    from paper_2604_26209_b200 import binding as B
    g = synth.Geom(Hq=2, Hkv=1, D=64, rope_theta=10000.0, sm_scale=0.125, suffix_cap=4)
    odd, host = torch.zeros(8, 8, device="cuda").t()[:, 1:], torch.zeros(1)
    calls = B._calls()
    lib = B.load()
    for name in calls.ENTRIES:
        kinds = getattr(lib, name).argtypes[1:-1]                # without the geometry and the stream
        pointers = [i for i, k in enumerate(kinds) if k is C.c_void_p]
        assert len(pointers) >= 4
        for i in pointers:
            for bad in (odd, host):
                with pytest.raises(AssertionError):
                    getattr(calls, name)(g, *[bad if j == i else None if j in pointers else 0 for j in range(len(kinds))])
