"""The conjugate-gradient solver on rods, on both sides of the edge lengths at which
it changes from the V-cycle to the diagonal, against the oracle's sparse direct
solve; the iterations tell which of the two ran."""
import numpy as np
import pytest

from oracle import ek_oracle as O
from test_gpu_krylov import rel, solve

pytestmark = pytest.mark.gpu

# (nz, ny, nx): does it take the diagonal
SHAPES = [((63, 6, 6), False), ((64, 6, 6), True), ((5, 5, 64), True), ((3, 63, 4), False), ((100, 1, 1), True),
          ((1, 8, 1), True), ((1, 2, 12), True), ((2, 2, 12), False), ((7, 8, 64), False)]


@pytest.mark.parametrize("shape,diagonal", SHAPES)
@pytest.mark.parametrize("held", [True, False])
def test_rods_against_the_oracle(gpu_lib, shape, diagonal, held):
    # as in test_gpu_krylov_levels.py
    rng = np.random.default_rng(13)
    eps = np.exp(0.5 * rng.normal(size=shape))
    q = rng.normal(size=shape)
    fixed = pf = None
    if held:
        fixed = np.zeros(shape, dtype=bool)
        fixed.ravel()[0] = True
        pf = np.where(fixed, 1.0, 0.0)
    phi, it, res = solve(gpu_lib, q, eps=eps, fixed=fixed, phi_fixed=pf)
    assert res <= 1e-13
    assert (it % 10 == 0) >= diagonal  # the diagonal's iterations come in tens
    assert rel(phi, O.poisson_dielectric(q, 0.7, eps=eps, fixed=fixed, phi_fixed=pf)) <= 1e-9
