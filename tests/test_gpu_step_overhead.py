"""What lbm_step(2) costs the host does not grow with the grid's rows: how a
grid would be cut into bands for the two-step kernel is settled when the
instance is made.  The two grids have the same cells and take the same two
single-step launches."""
import time

import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu


def enqueue_us(shape, calls=100, bursts=40):
    """The fastest burst's mean time of a call, the queue empty before it."""
    from paper_1608_06345_gb300 import lbm
    s = lbm.Solver(0, 1.4, 0.6, 0.7, shape, prec=lbm.LBM_F32)
    s.init(*li.random_fields(shape[0] * shape[1], 2, seed=1, u_amp=0.02))
    best = float("inf")
    for _ in range(bursts):
        s.sync()
        t = time.perf_counter()
        for _ in range(calls):
            s.step(2)
        best = min(best, time.perf_counter() - t)
    s.close()
    return 1e6 * best / calls


def test_step_time_does_not_grow_with_the_rows():
    few, many = enqueue_us((600, 4)), enqueue_us((4, 600))
    # a search over the bands on every call took 2 us more (3.8 and 5.9 us);
    # without one the two were within 4% of each other
    assert many < 1.3 * few, (few, many)
