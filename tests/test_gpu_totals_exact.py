"""Totals of FP32 and 16-bit storage against exact sums (math.fsum of the
stored values), on the fields that a compensated FP32 sum finds hardest:
uniform ones, where every thread makes the same rounding errors and nothing
averages out.  lbm_conserved_noalloc takes any planes; 4096 cells give every
thread its longest run.  Also the 16-bit decode, and deviations from a
reference state, whose sums cancel.

Tolerance: 2e-15 of the mass (momentum) and of the energy, that of the random
fields in tests/test_gpu_totals.py: the FP64 additions that follow the exact
group sums are a few dozen, each rounding by 2^-53."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 2e-15
GAMMA = 1.3  # delta = 4.67 in 2D, 3.67 in 3D


def lattice(lbm, lat):
    c, w, r = lbm.lbm_lattice_table(lat)
    return c.astype(float), np.asarray(w), r


def equilibrium(c, w, r, rho, u, T):
    """Second-order populations of a uniform state: values of the right sizes."""
    xi, D = r * c, c.shape[1]
    s, x2 = xi @ u, (xi ** 2).sum(1)
    g = w * rho * (1 + s + (s * s - u @ u + (T - 1) * (x2 - D)) / 2)
    return g, 0.5 * (2 / (GAMMA - 1) - D) * T * g


def check(got, g, h, c, r, N, rho0=0.0, T0=1.0):
    """got against N times the exact sums of one cell's stored g and h."""
    D = c.shape[1]
    delta = 2 / (GAMMA - 1) - D
    e = [0.5 * r * r * a * b for a, b in zip((c ** 2).sum(1), g)]
    ref = [N * math.fsum([rho0, *g])]
    ref += [r * N * math.fsum(a * b for a, b in zip(c[:, k], g)) for k in range(D)]
    ref += [N * math.fsum([rho0 * 0.5 * (D + delta) * T0, *e, *h])]
    scale = np.array([ref[0]] * (1 + D) + [ref[-1]])
    err = (got - np.array(ref)) / scale
    assert np.all(np.abs(err) <= TOL), err


@pytest.mark.parametrize("lat", [0, 1])
@pytest.mark.parametrize("seed", range(6))
@pytest.mark.parametrize("N", [4096, 13])  # whole runs of quads; quads and a remainder
def test_uniform_planes_sum_exactly(lat, seed, N):
    import torch

    from paper_1608_06345_gb300 import lbm
    c, w, r = lattice(lbm, lat)
    rng = np.random.default_rng(seed)
    g, h = equilibrium(c, w, r, rng.uniform(0.5, 2), rng.uniform(-0.08, 0.08, c.shape[1]), rng.uniform(0.8, 1.2))
    q = torch.tensor(np.concatenate([g, h]).astype(np.float32))
    stride = 4096
    state = q[:, None].expand(-1, stride).contiguous().cuda()
    got = lbm.lbm_conserved_noalloc(lat, lbm.LBM_F32, GAMMA, state, N, stride, rho0=-1.0)
    v = q.double().numpy()
    check(got, v[: len(w)], v[len(w):], c, r, N)


# runs of several quads of cells per thread; then the cells at which the
# blocks of 64 threads end (launch_conserve_t)
@pytest.mark.parametrize("lat,shape,prec", [(0, (2048, 1900), 1), (1, (160, 160, 40), 1), (0, (1024, 256), 1),
                                            (0, (5, 52429), 1), (0, (256, 256), 0), (0, (65537, 1), 0)])
def test_uniform_instance_sums_exactly(lat, shape, prec):
    import torch

    from paper_1608_06345_gb300 import lbm
    c, w, r = lattice(lbm, lat)
    N, D = math.prod(shape), len(shape)
    s = lbm.Solver(lat, GAMMA, 0.6, 0.7, shape, prec=prec, rho0=-1.0)
    u = torch.tensor([0.031, -0.017, 0.011][:D], dtype=torch.float64)[:, None].expand(-1, N).contiguous().cuda()
    s.init(torch.full((N,), 0.83, dtype=torch.float64, device="cuda"), u,
           torch.full((N,), 1.07, dtype=torch.float64, device="cuda"))
    got = s.conserved()
    ps = -(-N // 64) * 64
    v = s.mem.view(torch.float64 if prec == 0 else torch.float32)[: 2 * len(w) * ps].reshape(-1, ps)[:, 0].double().cpu().numpy()
    s.close()
    check(got, v[: len(w)], v[len(w):], c, r, N)


@pytest.mark.parametrize("prec", [2, 3])
@pytest.mark.parametrize("lat", [0, 1])
def test_16bit_pairs_are_decoded_and_summed(lat, prec):
    """Random stored pairs of FP16 or BF16: the decode is one FP32 product with
    the group's scale (gref, hscale) each."""
    import torch

    from paper_1608_06345_gb300 import lbm
    c, w, r = lattice(lbm, lat)
    Q, D, N, stride = len(w), c.shape[1], 5003, 5004
    rho0, T0 = 0.9, 1.1
    x2, th, delta = r * r * (c ** 2).sum(1), T0 - 1, 2 / (GAMMA - 1) - D
    gref = w * rho0 * (1 + (0.5 * th * (x2 - D) + 0.125 * th * th * (x2 * x2 - 2 * (D + 2) * x2 + D * (D + 2))))
    scale = torch.tensor(np.stack([gref, 0.5 * delta * T0 * gref], 1)).float().cuda()
    gen = torch.Generator(device="cuda").manual_seed(lat * 10 + prec)
    pairs = (0.05 * torch.randn((Q, stride, 2), generator=gen, device="cuda")).to(
        torch.float16 if prec == 2 else torch.bfloat16)
    got = lbm.lbm_conserved_noalloc(lat, prec, GAMMA, pairs, N, stride, rho0=rho0, T0=T0)
    q = (pairs[:, :N].float() * scale[:, None, :]).double().cpu().numpy()
    g = [math.fsum(x) for x in q[:, :, 0]]
    h = [math.fsum(x) for x in q[:, :, 1]]
    check(got, np.array(g) / N, np.array(h) / N, c, r, N, rho0, T0)


@pytest.mark.parametrize("lat,shape", [(0, (333, 5)), (1, (17, 9, 8))])
def test_deviation_storage_sums_exactly(lat, shape):
    """FP32 deviations from (rho0, T0): terms of both signs that cancel."""
    import lbm_inputs as li
    from paper_1608_06345_gb300 import lbm
    c, w, r = lattice(lbm, lat)
    N = math.prod(shape)
    s = lbm.Solver(lat, GAMMA, 0.6, 0.7, shape, prec=lbm.LBM_F32, rho0=0.9, T0=1.1)
    s.init(*li.random_fields(N, len(shape), seed=7, u_amp=0.02))
    s.step(2)
    raw = np.zeros(lbm.lbm_raw_state_bytes(s.h), dtype=np.uint8)
    lbm.lbm_get_state(s.h, raw)
    q = raw.view(np.float32).reshape(2 * len(w), N).astype(np.float64)
    got = s.conserved()
    s.close()
    g = [math.fsum(x) for x in q[: len(w)]]
    h = [math.fsum(x) for x in q[len(w):]]
    check(got, np.array(g) / N, np.array(h) / N, c, r, N, 0.9, 1.1)
