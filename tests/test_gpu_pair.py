"""Two steps per launch (large D2Q37 FP32 grids) against one launch per step
(lbm_set_graph_steps(h, 0)): the fields are equal bit for bit.  The grids are
the smallest that take the two-step way, with a last strip and bands of every
kind: strips of 119 and 120 columns, one strip, strips of the full 122 with
one band of a few rows, both boundary kinds on both axes, odd step counts,
graphs whose length is and is not a multiple of four, reference states other
than 1.  Each run is repeated, since a fault in the order of the waits would
show only now and then."""
import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu

CASES = [
    # shape, bc, steps, graph steps, rho0, T0
    ((1300, 700), (0, 0), 7, 64, 0.0, 0.0),
    ((2999, 300), (1, 0), 4, 64, 0.9, 1.1),
    ((122, 9000), (0, 1), 6, 64, -1.0, 0.0),
    ((18500, 41), (1, 1), 5, 64, 1.2, 0.8),
    ((1301, 701), (0, 1), 13, 6, 0.0, 0.0),
    ((1300, 700), (1, 0), 17, 8, 0.0, 0.0),
]


def fields_after(shape, bc, steps, graph, rho0, T0, fields):
    import torch

    from paper_1608_06345_gb300 import lbm
    N = shape[0] * shape[1]
    s = lbm.Solver(0, 1.4, 0.7, 0.6, shape, bc=bc, prec=lbm.LBM_F32, rho0=rho0, T0=T0)
    lbm.lbm_set_graph_steps(s.h, graph)
    s.init(*fields)
    s.step(steps)
    assert lbm.lbm_steps_done(s.h) == steps
    out = [torch.empty(n, dtype=torch.float64, device="cuda") for n in (N, 2 * N, N)]
    s.moments_device(*out)
    s.sync()
    s.close()
    return out


@pytest.mark.parametrize("shape,bc,steps,graph,rho0,T0", CASES)
def test_two_steps_per_launch_equal_single_steps(shape, bc, steps, graph, rho0, T0):
    import torch
    fields = li.random_fields(shape[0] * shape[1], 2, seed=sum(shape))
    ref = fields_after(shape, bc, steps, 0, rho0, T0, fields)
    for _ in range(4):
        got = fields_after(shape, bc, steps, graph, rho0, T0, fields)
        for a, b in zip(got, ref):
            assert torch.equal(a, b)


def test_a_nonfinite_cell_is_reported_from_either_of_the_two_steps():
    from paper_1608_06345_gb300 import lbm
    shape = (1300, 700)
    rho, u, T = li.uniform_fields(shape[0] * shape[1], 2)
    rho[shape[0] * 350 + 600] = np.nan
    for steps in (2, 3):
        s = lbm.Solver(0, 1.4, 0.6, 0.6, shape, prec=lbm.LBM_F32)
        s.init(rho, u, T)
        s.step(steps)
        with pytest.raises(lbm.LbmError) as ei:
            s.sync()
        assert ei.value.code == lbm.LBM_ENONFINITE
        s.close()
