"""lbm_conserved against the sums of the raw state's values, taken exactly
(math.fsum) on the host.  FP32 and 16-bit storage sum 16-byte loads of four
cells with their rounding errors kept, cells past the last four one by one,
and runs that are not finite again in FP64: sizes below and above one block
and one run, each remainder of four cells, and states holding infinities,
NaN and values whose FP32 sum overflows."""
import math

import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu


def values(lbm, s):
    """The stored deviations (g, h) as exact doubles, each (Q, N)."""
    raw = np.zeros(lbm.lbm_raw_state_bytes(s.h), dtype=np.uint8)
    lbm.lbm_get_state(s.h, raw)
    if s.prec == lbm.LBM_F64:
        q = raw.view(np.float64).reshape(2 * s.Q, s.N)
    else:
        q = raw.view(np.float32).reshape(2 * s.Q, s.N).astype(np.float64)
    return q[: s.Q], q[s.Q:]


def exact_totals(lbm, s, gamma):
    g, h = values(lbm, s)
    c, _, r = lbm.lbm_lattice_table(s.lattice)
    rows = [g, *(r * c[:, a:a + 1] * g for a in range(s.D)), 0.5 * r * r * (c ** 2).sum(1)[:, None] * g]
    t = np.array([math.fsum(x.ravel()) for x in rows])
    t[-1] += math.fsum(h.ravel())
    return t


# one cell, remainders 0..3 of four cells, more than a block of quads, more
# than one run of 16 cells per thread (912 x 256 threads x 16 cells)
SIZES_2D = [(1, 1), (5, 1), (37, 2), (333, 5), (4099, 1), (2051, 1861)]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("lat,shape", [(0, n) for n in SIZES_2D] + [(1, (7, 3, 5)), (1, (64, 33, 9))])
def test_totals_are_the_sums_of_the_state(lat, shape, prec):
    from paper_1608_06345_gb300 import lbm
    N, D = int(np.prod(shape)), len(shape)
    s = lbm.Solver(lat, 1.4, 0.6, 0.7, shape, prec=prec, rho0=-1.0)  # whole storage: nothing is added on the host
    s.init(*li.random_fields(N, D, seed=N))
    s.step(2)
    got, ref = s.conserved(), exact_totals(lbm, s, 1.4)
    s.close()
    # every term is exact to its last bit and the partial sums are FP64: a few
    # units of 2^-53 of the mass (momentum) and of the energy
    scale = np.array([ref[0]] * (1 + D) + [ref[-1]])
    assert np.all(np.abs(got - ref) <= 2e-15 * scale), (got, ref)


@pytest.mark.parametrize("value,kind", [(np.inf, "inf"), (np.nan, "nan"), (3e38, "large")])
def test_totals_of_a_state_that_does_not_sum_in_fp32(value, kind):
    from paper_1608_06345_gb300 import lbm
    shape = (301, 3)
    s = lbm.Solver(0, 1.4, 0.6, 0.7, shape, prec=1, rho0=-1.0)
    s.init(*li.random_fields(903, 2, seed=3))
    raw = np.zeros(lbm.lbm_raw_state_bytes(s.h), dtype=np.uint8)
    lbm.lbm_get_state(s.h, raw)
    q = raw.view(np.float32).reshape(74, 903)
    q[0, 7] = value      # the rest velocity: mass only
    q[0, 8] = value
    q[1, 900] = 1.0      # (1, 0), a cell of the remainder
    lbm.lbm_set_state(s.h, raw)
    got = s.conserved()
    s.close()
    if kind == "inf":
        assert got[0] == np.inf and np.all(np.isfinite(got[1:3]))
    elif kind == "nan":
        assert np.isnan(got[0]) and np.all(np.isfinite(got[1:3]))
    else:
        assert abs(got[0] / (2 * float(np.float32(3e38))) - 1) < 1e-15
