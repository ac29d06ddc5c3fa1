"""A finite-difference step of a thin grid takes about as long as one of the
same number of cells in a compact one: the tile kernel, most of whose threads
would have no cell there, leaves it to the row kernel (launch_step_fd_t)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def us_per_step(lat, prec, shape, steps=50):
    import torch

    from paper_1608_06345_gb300 import lbm
    N, D = int(np.prod(shape)), len(shape)
    s = lbm.Solver(lat, 1.4, 0.8, 0.8, shape, prec=prec)
    one = torch.ones(N, dtype=torch.float64, device="cuda")
    s.init(one, torch.zeros(D * N, dtype=torch.float64, device="cuda"), one)
    best = float("inf")
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        s.step_fd(steps, 0.03)
        b.record()
        b.synchronize()
        best = min(best, 1e3 * a.elapsed_time(b) / steps)
    s.close()
    return best


@pytest.mark.parametrize("lat,prec,thin,compact", [
    (1, 1, (20000, 1, 1), (200, 10, 10)),  # the tile kernel took 194 us
    (1, 2, (20000, 1, 1), (200, 10, 10)),  # 171
    (1, 0, (20000, 1, 1), (320, 63, 1)),   # 563
    (0, 2, (100000, 1), (1000, 100)),      # 26
])
def test_thin_grids_are_not_slower(lat, prec, thin, compact):
    t, c = us_per_step(lat, prec, thin), us_per_step(lat, prec, compact)
    assert t <= 1.5 * c, (t, c)
