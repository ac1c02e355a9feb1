"""Native marshalling of the per-step calls: what it refuses, before anything reaches the library (no GPU needed)."""
import numpy as np
import pytest
import torch

from paper_2604_26209_b200 import binding, synth

GEOM = synth.Geom(Hq=4, Hkv=1, D=64, rope_theta=10000.0, sm_scale=0.125, suffix_cap=4)


def test_every_step_call_is_marshalled_natively():
    host = binding._calls()
    assert set(host.ENTRIES) == {n for n in binding.EXPORTS if n.startswith("hpd_")} - {
        "hpd_strerror", "hpd_last_cuda_error", "hpd_workspace_bytes"}


@pytest.mark.parametrize("args,error", [
    ((GEOM, 1, torch.zeros(4), None, None, None), AssertionError),       # a tensor that is not on the device
    ((GEOM, 1, [0], None, None, None), TypeError),                       # not a tensor
    ((GEOM, 1.0, None, None, None, None), TypeError),                    # not an integer
    ((GEOM, 1, None, None, None), TypeError),                            # an argument too few
    ((object(), 1, None, None, None, None), AttributeError),             # not a geometry
])
def test_refused_arguments(args, error):
    with pytest.raises(error):
        binding._calls().hpd_rope(*args)


@pytest.mark.parametrize("n", [0, False, np.int32(0), np.int64(0), torch.tensor(0)])
def test_sizes_may_be_any_integer(n):
    """Whatever has an integer value passes, as it does through ctypes: the call gets as far as the current stream."""
    if torch.cuda.is_available():
        assert binding._calls().hpd_rope(GEOM, n, None, None, None, None) == 0
    else:
        with pytest.raises(RuntimeError):
            binding._calls().hpd_rope(GEOM, n, None, None, None, None)
