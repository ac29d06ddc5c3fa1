"""The FP64 step takes relaxation times up to the largest double as the oracle
takes them (its constants carry 1 / tau_f in the weights and tau_f in the
factor of h)."""
import numpy as np
import pytest

import lbm_inputs as li
from tests.parity import TOL, assert_parity, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau_f", [40.0, 1e6, 1e12, 1e17, 1e305, 1.7e308])
@pytest.mark.parametrize("lat,shape", [(0, (32, 8)), (1, (12, 5, 4))])
def test_large_relaxation_times_match_the_oracle(lat, shape, tau_f):
    from paper_1608_06345_gb300 import lbm
    D = len(shape)
    fields = li.random_fields(int(np.prod(shape)), D, seed=3, u_amp=0.02)
    ref, _ = run_oracle(lat, 1.4, tau_f, 0.7, shape, (0,) * D, fields, 5)
    s = lbm.Solver(lat, 1.4, tau_f, 0.7, shape, prec=lbm.LBM_F64)
    s.init(*fields)
    s.step(5)
    got = s.moments()
    s.close()
    assert_parity(got, ref, 1.4, TOL["f64"])
