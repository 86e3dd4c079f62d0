"""The momentum exchange of S4 takes the nodes next to a particle from a list per
warp: the largest sphere of a box (a widened box larger than the lattice), the
smallest, one over the periodic corner, one and several particles, flat and odd
boxes, in both forms against the FP64 oracle."""
import numpy as np
import pytest

from oracle import ek_oracle as O
from pairs import TOL, compare, make_pair

pytestmark = pytest.mark.gpu

CASES = {
    "largest": ((16, 16, 16), [((8.3, 7.6, 8.1), 5.0)]),
    "smallest": ((16, 9, 12), [((8.3, 4.6, 6.1), 1.0)]),
    "corner": ((18, 16, 24), [((0.1, 15.9, 23.8), 4.0)]),
    "several": ((32, 16, 18), [((6.2, 8.1, 9.3), 4.0), ((17.1, 7.9, 9.0), 3.0), ((25.0, 8.4, 8.7), 2.5)]),
}


def pair(ek, name, flags):
    shape, spheres = CASES[name]
    case = dict(shape=shape, nu=1.0 / 6.0, rho0=1.0, bjerrum=0.7, valence=(1, -1), D=(0.3, 0.3), bulk=(1e-3, 1e-3),
                E=(0.004, -0.002, 0.003), rho_p=2.0,
                particles=[dict(pos=c, radius=R, charge=-6.0) for c, R in spheres])
    n = len(spheres)
    return make_pair(ek, case, flags=flags, vel=[(0.02, -0.01, 0.01)] * n, omega=[(0.001, 0.002, -0.001)] * n)


@pytest.mark.parametrize("name", sorted(CASES))
def test_links_fp64(gpu_lib, name):
    o, s = pair(gpu_lib, name, O.PV | O.NEUTRALIZE)
    o.step(3)
    s.step(3)
    compare(gpu_lib, o, s, tol=TOL)


@pytest.mark.parametrize("name", sorted(CASES))
def test_links_fp32(gpu_lib, name):
    o, s = pair(gpu_lib, name, O.PV | O.NEUTRALIZE | 16)
    o.step(3)
    s.step(3)
    for p, q in zip(s.get_particles(), o.particles):
        # FP32 populations and sums against FP64, as in the field comparisons
        assert np.max(np.abs(p["pos"] - q.pos)) < 1e-6
        assert np.max(np.abs(p["vel"] - q.vel)) < 1e-3 * np.max(np.abs(q.vel))
