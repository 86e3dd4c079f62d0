"""The level structure of the conjugate-gradient solver's preconditioner: boxes
with odd edges, edges too short to halve, edges of 1 and 2, red-black and
Jacobi levels mixed, a single level, against the oracle's sparse direct solve;
with fixed planes, an electrode and without any fixed node."""
import numpy as np
import pytest

from oracle import ek_oracle as O
from test_gpu_krylov import rel, solve

pytestmark = pytest.mark.gpu

# (nz, ny, nx)
SHAPES = [(8, 8, 8), (9, 16, 7), (13, 13, 13), (40, 6, 50), (1, 16, 33), (2, 24, 18), (7, 7, 7),
          (34, 12, 66), (20, 4, 3)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("held", [True, False])
def test_levels_against_the_oracle(gpu_lib, shape, held):
    # the residual falls to 1e-13 of the charge's; the operator's condition is
    # about the square of the longest edge (4e3) times the permittivity's
    # spread (10): errors up to some 1e-9
    rng = np.random.default_rng(11)
    eps = np.exp(0.5 * rng.normal(size=shape))
    q = rng.normal(size=shape)
    fixed = pf = None
    if held:
        z, y, x = np.meshgrid(*(np.arange(n) for n in shape), indexing="ij")
        fixed = (x == 0) | ((x == shape[2] - 1) & (y < shape[1] // 2))
        pf = np.where(x == 0, 1.0, -0.5)
    phi, it, res = solve(gpu_lib, q, eps=eps, fixed=fixed, phi_fixed=pf)
    assert res <= 1e-13
    ref = O.poisson_dielectric(q, 0.7, eps=eps, fixed=fixed, phi_fixed=pf)
    if held:
        assert np.array_equal(phi[fixed], pf[fixed])
    assert rel(phi, ref) <= 1e-9
