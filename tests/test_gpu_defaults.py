"""The default launch shape picks a kernel by the grid's size (launch_impl.cuh).
All the kernels it picks from give the same bits: every FP64 shape (the split
kernels sum the moments in the order of the others), and the D3Q107 shapes of
FP32 and 16-bit storage that differ only in their block width.  The batched
pool, which has one kernel per storage, gives the bits of a lone instance on
either side of each threshold."""
import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu


def run(lat, prec, shape, bc, fields, index, steps=7):
    from paper_1608_06345_gb300 import lbm
    s = lbm.Solver(lat, 1.4, 0.6, 0.7, shape, bc=bc, prec=prec)
    lbm.lbm_set_shape(s.h, index)
    s.init(*fields)
    s.step(steps)
    out = s.moments()
    s.close()
    return out


# lattice, prec, shape (rows below, at and above the widths and the FP64 threshold of 304 blocks of 32 cells), indices
CASES = [
    (0, 0, (45, 3), (1, 0), range(5)),
    (0, 0, (1000, 10), (1, 0), range(5)),
    (1, 0, (33, 8, 9), (0, 1, 0), range(4)),
    (1, 1, (20, 8, 9), (0, 1, 0), (0, 1, 2, 6)),
    (1, 1, (97, 7, 8), (1, 0, 1), (0, 1, 2, 6)),
    (1, 1, (128, 5, 4), (0, 0, 0), (0, 1, 2, 6)),
    (1, 2, (97, 7, 8), (1, 0, 1), (0, 1, 2, 6)),
    (1, 3, (40, 9, 7), (0, 0, 0), (0, 1, 2, 6)),
]


@pytest.mark.parametrize("lat,prec,shape,bc,indices", CASES)
def test_shapes_of_one_rounding_give_the_same_bits(lat, prec, shape, bc, indices):
    fields = li.random_fields(int(np.prod(shape)), len(shape), seed=sum(shape), u_amp=0.02)
    ref = run(lat, prec, shape, bc, fields, 0)
    for k in indices:
        for a, b in zip(run(lat, prec, shape, bc, fields, k), ref):
            assert np.array_equal(a, b), k


@pytest.mark.parametrize("lat,prec,shapes", [(0, 0, [(300, 4), (3000, 5)]), (1, 0, [(40, 5, 6), (9, 8, 7)]),
                                             (1, 2, [(40, 5, 6), (100, 8, 7)]), (1, 1, [(33, 8, 9), (130, 4, 5)])])
def test_pool_gives_the_bits_of_a_lone_instance(lat, prec, shapes):
    from paper_1608_06345_gb300 import lbm
    D = len(shapes[0])
    pool = lbm.Pool(lat, prec, budget_bytes=256 << 20, max_instances=4, bundle_steps=4)
    jobs = []
    for shape in shapes:
        fields = li.random_fields(int(np.prod(shape)), D, seed=sum(shape), u_amp=0.02)
        bc = (1,) + (0,) * (D - 1)
        jobs.append((shape, bc, fields, pool.submit(1.4, 0.6, 0.7, shape, bc, fields, 7)))
    pool.run(2)
    pool.sync()
    for shape, bc, fields, ticket in jobs:
        rc, got = pool.result(ticket, int(np.prod(shape)))
        for a, b in zip(got, run(lat, prec, shape, bc, fields, 0)):
            assert np.array_equal(a, b)
    pool.close()


@pytest.mark.parametrize("prec,shape", [(1, (33, 5)), (1, (127, 3)), (1, (1, 40)), (2, (1003, 431)), (3, (433, 1001))])
def test_cells_in_memory_order_give_the_bits_of_the_pool(prec, shape):
    """Rows that are no multiple of 32 cells run as one flat range of cells
    (16-bit storage: off the sectors and larger than L2); the pool works row
    by row."""
    from paper_1608_06345_gb300 import lbm
    fields = li.random_fields(int(np.prod(shape)), 2, seed=sum(shape), u_amp=0.02)
    pool = lbm.Pool(0, prec, budget_bytes=256 << 20, max_instances=2, bundle_steps=5)
    ticket = pool.submit(1.4, 0.6, 0.7, shape, (1, 0), fields, 5)
    pool.run(1)
    pool.sync()
    rc, got = pool.result(ticket, int(np.prod(shape)))
    pool.close()
    for a, b in zip(got, run(0, prec, shape, (1, 0), fields, 0, steps=5)):
        assert np.array_equal(a, b)
