"""The small levels of the conjugate-gradient solver's V-cycle run in one cluster of
as many thread blocks as the device can place: fewer give the same result."""
import numpy as np
import pytest

from test_gpu_krylov import solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(24, 40, 32), (17, 26, 33)])
def test_smaller_clusters_give_the_same_solution(gpu_lib, shape):
    ek = gpu_lib
    rng = np.random.default_rng(12)
    eps = np.exp(0.5 * rng.normal(size=shape))
    q = rng.normal(size=shape)
    fixed = np.zeros(shape, dtype=bool)
    fixed[0] = True
    try:
        got = []
        for n in (0, 8, 4, 3, 2, 1):
            ek.debug_cluster_limit(n)
            got.append(solve(ek, q, eps=eps, fixed=fixed, phi_fixed=fixed.astype(np.float64)))
    finally:
        ek.debug_cluster_limit(0)
    for phi, it, res in got[1:]:
        assert np.array_equal(phi, got[0][0]) and it == got[0][1] and res == got[0][2]
