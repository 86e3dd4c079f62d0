"""What the multigrid solve converges to, beyond its tolerance."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LB = 0.7


def solve(ek, q, shape, tol, max_cycles):
    import torch
    nx, ny, nz = shape
    qd = torch.tensor(q.ravel(), device="cuda", dtype=torch.float64)
    scratch = torch.empty(ek.poisson_mg_scratch_bytes(shape), dtype=torch.uint8, device="cuda")
    phi = torch.empty_like(qd)
    cycles, res = ek.poisson_solve_mg(qd, phi, shape, LB, scratch, tol=tol, max_cycles=max_cycles)
    return phi.cpu().numpy().reshape(nz, ny, nx), cycles, res


@pytest.mark.parametrize("shape,axis", [((128, 32, 32), 2), ((32, 128, 32), 1), ((32, 32, 128), 0)])
def test_the_longest_wave_has_no_bias(gpu_lib, shape, axis):
    """The potential's part along the longest wave of the box, cos(2 pi x / 128),
    against its value 4 pi l_B q / lambda, lambda = 2 - 2 cos(2 pi / 128).  Noise of
    the wave's own size in the charge makes the nodes' roundings independent.

    A residual of 6 2^-54 phi left on half of the nodes changes the part by
    3 2^-54 / lambda = 6.9e-14 of itself.  Roundings of some 6 2^-53 phi a node add
    up at random over 131072 nodes: 7.6e-16.  The bound lies between them."""
    n = 128
    wave = np.cos(2.0 * np.pi * np.arange(n) / n).reshape([n if a == axis else 1 for a in range(3)])
    q = wave + np.random.default_rng(8).standard_normal(shape[::-1])
    phi, _, res = solve(gpu_lib, q, shape, tol=1e-16, max_cycles=30)
    assert res < 1e-12
    long = np.longdouble
    w = np.cos(2 * np.arccos(long(-1)) * np.arange(n).astype(long) / n).reshape(wave.shape)
    lam = 2 - 2 * np.cos(2 * np.arccos(long(-1)) / n)
    want = 4 * np.arccos(long(-1)) * long(LB) * (q.astype(long) * w).sum() / lam
    assert abs((phi.astype(long) * w).sum() / want - 1) < 1e-14


@pytest.mark.parametrize("shape", [(54, 54, 54), (162, 27, 32)])
def test_a_box_that_cannot_be_coarsened_takes_one_cycle(gpu_lib, shape):
    """Also below the residual that rounding leaves, eps 12 max|phi| / max|b| and more:
    the FFT solves the whole problem, and again would give the same."""
    q = np.random.default_rng(9).standard_normal(shape[::-1])
    first, cycles, res = solve(gpu_lib, q, shape, tol=1e-9, max_cycles=50)
    assert cycles == 1 and res < 1e-9
    again, cycles, res = solve(gpu_lib, q, shape, tol=1e-17, max_cycles=50)
    assert cycles == 1 and 1e-17 < res < 1e-9
    assert np.array_equal(first, again)
