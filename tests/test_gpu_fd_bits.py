"""The row and the tile kernel of the finite-difference step give the same
bits.  Grids of few tiles take the row kernel, larger ones the tile kernel
(launch_step_fd_t), so a small periodic grid and the same fields repeated
along its last axis run one each, and every copy must equal the small grid's
result."""
import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu

CASES = [
    # lattice, prec, small grid, boundaries, copies (tiles of the small and the repeated grid; the line lies at)
    (1, 0, (33, 20, 20), (1, 0, 0), 5),  # 75 and 375 tiles of 16 x 4 x 4 (two per SM)
    (1, 0, (33, 21, 19), (0, 1, 0), 6),  # ragged in y and z: 90 and 522
    (1, 1, (33, 20, 6), (0, 1, 0), 10),  # 3960 and 39600 cells (200 per SM)
    (1, 2, (33, 20, 6), (1, 0, 0), 10),
    (1, 3, (20, 17, 7), (1, 1, 0), 14),  # 2380 and 33320
    (0, 2, (100, 40), (1, 0), 30),       # 20 and 600 of 32 x 8 (three per SM)
    (0, 3, (75, 41), (0, 0), 40),        # 18 and 615
]


def run(lat, prec, shape, bc, fields):
    from paper_1608_06345_gb300 import lbm
    s = lbm.Solver(lat, 1.4, 0.8, 0.7, shape, bc=bc, prec=prec)
    s.init(*fields)
    s.step_fd(4, 0.03)
    out = s.moments()
    s.close()
    return out


@pytest.mark.parametrize("lat,prec,shape,bc,copies", CASES)
def test_row_and_tile_kernel_give_the_same_bits(lat, prec, shape, bc, copies):
    N = int(np.prod(shape))
    fields = li.random_fields(N, len(shape), seed=sum(shape), u_amp=0.02, rho_amp=0.02, T_amp=0.02)
    small = run(lat, prec, shape, bc, fields)
    large = run(lat, prec, shape[:-1] + (shape[-1] * copies,), bc,
                tuple(np.concatenate([f] * copies, axis=-1) for f in fields))
    for a, b in zip(small, large):
        assert np.array_equal(np.concatenate([a] * copies, axis=-1), b)
