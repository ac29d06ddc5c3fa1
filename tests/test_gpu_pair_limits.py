"""The two-step kernel's limits: a wait that gives up ends the run in
LBM_ETIMEOUT and leaves the GPU usable, and grids whose element indices need
64 bits (74 planes of more than 2^32 elements) give the bits of single steps."""
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu


def solver(shape, prec=1):
    from paper_1608_06345_gb300 import lbm
    s = lbm.Solver(0, 1.4, 0.7, 0.6, shape, prec=prec)
    s.init(*li.random_fields(shape[0] * shape[1], 2, seed=2, u_amp=0.02))
    return s


@pytest.mark.parametrize("steps", [2, 130])  # a launch; replays of a graph
def test_a_wait_that_gives_up_is_reported(steps):
    from paper_1608_06345_gb300 import lbm
    s = solver((1300, 700))
    assert lbm.lbm_step_info(s.h)[2] == 2
    s.step(steps)
    s.sync()  # the default limit is not reached
    lbm.lbm_set_wait_limit(s.h, 0)
    s.step(steps)
    for call in (s.sync, s.moments, s.conserved):
        with pytest.raises(lbm.LbmError) as err:
            call()
        assert err.value.code == lbm.LBM_ETIMEOUT
    s.close()
    other = solver((200, 6))  # the context goes on
    other.step(3)
    other.sync()
    other.close()


def test_the_limit_is_checked():
    from paper_1608_06345_gb300 import lbm
    s = solver((20, 5))
    with pytest.raises(lbm.LbmError) as err:
        lbm.lbm_set_wait_limit(s.h, -1)
    assert err.value.code == lbm.LBM_EINVAL
    s.close()


def test_indices_beyond_32_bits():
    import torch

    from paper_1608_06345_gb300 import lbm
    shape = (7711, 7601)
    N = shape[0] * shape[1]
    assert 74 * N >= 2 ** 32
    gen = torch.Generator(device="cuda").manual_seed(3)
    noise = 0.04 * torch.rand((4, N), generator=gen, device="cuda", dtype=torch.float64) - 0.02
    fields = 1 + noise[0], noise[1:3].contiguous(), 1 + noise[3]
    out = []
    for index in (0, 1):
        s = lbm.Solver(0, 1.4, 0.7, 0.6, shape, bc=(1, 0), prec=lbm.LBM_F32)
        lbm.lbm_set_shape(s.h, index)
        assert lbm.lbm_step_info(s.h)[2] == 2 - index
        s.init(*fields)
        s.step(3)
        q = [torch.empty(n, dtype=torch.float64, device="cuda") for n in (N, 2 * N, N)]
        s.moments_device(*q)
        s.sync()
        s.close()
        del s
        out.append(q)
    for a, b in zip(*out):
        assert torch.equal(a, b)
