"""The tiled finite-difference kernel against the oracle, on grids just large
enough to take it (launch_step_fd_t): ragged last tiles on every axis, both
boundary kinds on every axis, and each storage that uses it.  Tolerances are
those of tests/test_gpu_fd.py: the parity bars for FP64 and FP32, the stated
bounds for 16-bit storage."""
import numpy as np
import pytest

import lbm_inputs as li
from oracle import oracle as ora
from tests.parity import TOL, assert_parity

pytestmark = pytest.mark.gpu

P, ZG = ora.PERIODIC, ora.ZERO_GRADIENT
CASES = [
    # lattice, prec, shape, bc, steps, tolerance
    (1, 1, (37, 33, 45), (P, ZG, P), 4, TOL["f32"]),      # 3 x 5 x 12 tiles of 16 x 8 x 4
    (1, 1, (65, 31, 18), (ZG, P, ZG), 4, TOL["f32"]),
    (1, 2, (37, 33, 45), (ZG, P, P), 4, 2e-3),
    (1, 3, (33, 40, 29), (P, P, ZG), 4, 2e-2),
    (1, 0, (33, 41, 46), (ZG, P, ZG), 3, TOL["f64"]),     # 3 x 11 x 12 tiles of 16 x 4 x 4
    (0, 2, (517, 235), (P, ZG), 6, 5e-3),                 # 17 x 30 tiles of 32 x 8
    (0, 3, (1025, 113), (ZG, P), 6, 6e-2),
]


@pytest.mark.parametrize("lat,prec,shape,bc,steps,tol", CASES)
def test_tiled_fd_step_matches_the_oracle(lat, prec, shape, bc, steps, tol):
    from paper_1608_06345_gb300 import lbm
    D = len(shape)
    fields = li.random_fields(int(np.prod(shape)), D, seed=sum(shape), u_amp=0.02, rho_amp=0.02, T_amp=0.02)
    o = ora.Oracle(lat, 1.4, 0.8, 0.7, shape, bc=bc)
    o.init(*fields)
    o.step_fd(steps, 0.03)
    s = lbm.Solver(lat, 1.4, 0.8, 0.7, shape, bc=bc, prec=prec)
    s.init(*fields)
    s.step_fd(steps, 0.03)
    got = s.moments()
    s.close()
    assert_parity(got, o.moments(), 1.4, tol)
