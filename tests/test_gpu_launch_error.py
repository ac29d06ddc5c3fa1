"""A launch that the runtime refuses is reported by the call that made it and
by no other: the error is not left behind for the next launch's check."""
import ctypes

import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["step", "step_fd"])
def test_a_refused_launch_does_not_fail_the_next_call(call):
    import torch

    from paper_1608_06345_gb300 import lbm
    cuda = ctypes.CDLL("libcuda.so.1")
    s = lbm.Solver(0, 1.4, 0.7, 0.7, (40, 6), stream=torch.cuda.default_stream())
    s.init(*li.random_fields(240, 2, seed=4, u_amp=0.02))
    before = s.moments()
    # while a blocking stream is being captured, nothing may be launched into
    # the legacy default stream
    stream, graph = ctypes.c_void_p(), ctypes.c_void_p()
    assert cuda.cuStreamCreate(ctypes.byref(stream), 0) == 0
    assert cuda.cuStreamBeginCapture_v2(stream, 0) == 0
    try:
        with pytest.raises(lbm.LbmError) as err:
            getattr(s, call)(1)
    finally:
        cuda.cuStreamEndCapture(stream, ctypes.byref(graph))  # the refusal has ended the capture; the error says so
        cuda.cuStreamDestroy_v2(stream)
    assert err.value.code == lbm.LBM_ECUDA
    for a, b in zip(s.moments(), before):
        assert np.array_equal(a, b)
    s.close()
