"""What lbm_step runs (lbm_step_info) follows the chosen shape: index 0 takes
two steps per launch on large D2Q37 FP32 grids, an explicit index or graph
length 0 one; the table names the kernels that run, and the autotuner times
index 0 as it runs and none of its kernels twice."""
import numpy as np
import pytest

import lbm_inputs as li
from tests.test_gpu_pair import CASES as PAIR_CASES

pytestmark = pytest.mark.gpu


def solver(lat, shape, prec, **kw):
    from paper_1608_06345_gb300 import lbm
    s = lbm.Solver(lat, 1.4, 0.7, 0.6, shape, prec=prec, **kw)
    s.init(*li.random_fields(int(np.prod(shape)), len(shape), seed=1, u_amp=0.02))
    return s


@pytest.mark.parametrize("shape", sorted({c[0] for c in PAIR_CASES}) + [(607, 330), (1000, 340)])
def test_large_grids_go_two_steps_per_launch_unless_told_otherwise(shape):
    from paper_1608_06345_gb300 import lbm
    s = solver(0, shape, lbm.LBM_F32)
    assert lbm.lbm_step_info(s.h) == (10, 128, 2)
    lbm.lbm_set_shape(s.h, 1)
    assert lbm.lbm_step_info(s.h) == (0, 256, 1)
    s.step(5)
    one = s.moments()
    lbm.lbm_set_shape(s.h, 0)
    lbm.lbm_set_graph_steps(s.h, 0)
    assert lbm.lbm_step_info(s.h) == (0, 128, 1)
    lbm.lbm_set_graph_steps(s.h, 4)
    assert lbm.lbm_step_info(s.h) == (10, 128, 2)
    s.init(*li.random_fields(shape[0] * shape[1], 2, seed=1, u_amp=0.02))
    s.step(5)
    for a, b in zip(s.moments(), one):
        assert np.array_equal(a, b)
    s.close()


@pytest.mark.parametrize("lat,prec,shape,expected", [
    (0, 1, (300, 200), (0, 128, 1)), (0, 0, (1000, 4), (4, 32, 1)), (0, 0, (1000, 16), (0, 128, 1)),
    (1, 0, (20, 9, 8), (7, 32, 1)), (1, 1, (32, 9, 8), (3, 32, 1)), (1, 1, (100, 9, 8), (3, 128, 1)),
    (1, 1, (129, 9, 8), (3, 32, 1)), (1, 1, (190, 9, 8), (3, 64, 1)), (1, 2, (97, 9, 8), (6, 64, 1)),
    (1, 3, (96, 9, 8), (6, 32, 1))])
def test_index_0_is_picked_by_size(lat, prec, shape, expected):
    from paper_1608_06345_gb300 import lbm
    s = solver(lat, shape, prec)
    assert lbm.lbm_step_info(s.h) == expected
    s.close()


def test_the_table_names_the_kernels_of_large_grids():
    from paper_1608_06345_gb300 import lbm
    for lat, prec, shape in ((1, 0, (64, 30, 30)), (1, 1, (256, 30, 30)), (1, 2, (256, 30, 30)), (0, 0, (512, 256))):
        s = solver(lat, shape, prec)
        assert lbm.lbm_step_info(s.h)[:2] == lbm.lbm_shape_info(lat, prec, 0)
        k = 1
        while lbm.lbm_shape_info(lat, prec, k) is not None:
            lbm.lbm_set_shape(s.h, k)
            assert lbm.lbm_step_info(s.h)[:2] == lbm.lbm_shape_info(lat, prec, k)
            k += 1
        s.close()


def test_the_autotuner_times_what_lbm_step_runs():
    from paper_1608_06345_gb300 import autotune, lbm
    s = lbm.Solver(0, 1.4, 0.7, 0.6, (4096, 1024), prec=lbm.LBM_F32)  # two steps per launch are 1.2 times as fast
    lbm.lbm_set_shape(s.h, 2)
    import torch
    N = 4096 * 1024
    one = torch.ones(N, dtype=torch.float64, device="cuda")
    s.init(one, torch.zeros(2 * N, dtype=torch.float64, device="cuda"), one)
    rec = autotune.tune(s, reps=5, cache_path=None)
    assert (rec["index"], rec["stage"], rec["steps_per_launch"]) == (0, 10, 2)
    lbm.lbm_set_graph_steps(s.h, 0)
    single = autotune.tune(s, reps=5, cache_path=None)
    assert single["steps_per_launch"] == 1 and single["stage"] == 0
    assert rec["us_per_step"] < single["us_per_step"]
    s.close()
    # D3Q107 FP64: index 3 is index 0's kernel, which wins a tie
    s = solver(1, (32, 9, 8), lbm.LBM_F64)
    assert autotune.tune(s, reps=2, cache_path=None)["index"] != 3
    s.close()
