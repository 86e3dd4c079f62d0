"""S2 and S3 of both storage forms on the boxes where their 32 x 8 tiles and
plane segments can go wrong: narrower than a tile, one past it, ragged, flat and
deep, with one to four species, with and without partial volumes, walls across
the tiles and a sphere over the periodic seam, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import ek_oracle as O
from pairs import TOL, compare, make_pair, perm_to_oracle

pytestmark = pytest.mark.gpu

SHAPES = [(8, 9, 8), (36, 9, 27), (64, 8, 8), (54, 18, 12), (32, 16, 81)]
SPECIES = {1: (1,), 2: (1, -1), 3: (1, -1, 2), 4: (1, -1, 2, -2)}


def case(shape, K, sphere=False):
    # a sphere whose centre lies on the corner of the box
    parts = [dict(pos=(0.2, 0.3, shape[2] - 0.4), radius=2.5, charge=-6.0)] if sphere else []
    return dict(shape=shape, nu=1.0 / 6.0, rho0=1.0, bjerrum=0.7, valence=SPECIES[K],
                D=(0.2, 0.3, 0.15, 0.1)[:K], bulk=(1e-3,) * K, E=(0.004, -0.002, 0.003), particles=parts, rho_p=2.0)


def walls_of(shape):
    nx, ny, nz = shape
    w = np.zeros((nz, ny, nx), dtype=bool)
    w[0] = True
    w[:, ny // 2, : nx // 2] = True
    return w


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("K", [1, 2, 3, 4])
def test_fp64_tiles(gpu_lib, shape, K):
    o, s = make_pair(gpu_lib, case(shape, K), flags=O.PV, magic=3.0 / 16.0, walls=walls_of(shape),
                     g=(1e-5, 2e-5, -1e-5))
    o.step(3)
    s.step(3)
    compare(gpu_lib, o, s, tol=TOL)


@pytest.mark.parametrize("shape", [(12, 16, 18), (36, 12, 27), (64, 16, 12)])
@pytest.mark.parametrize("flags", [O.PV, 0])
def test_fp64_tiles_with_a_sphere_on_the_seam(gpu_lib, shape, flags):
    o, s = make_pair(gpu_lib, case(shape, 2, True), flags=flags, vel=[(0.03, -0.02, 0.05)], omega=[(1e-3, 0.0, 2e-3)])
    for _ in range(3):
        o.step(2)
        s.step(2)
        compare(gpu_lib, o, s, tol=TOL)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("K", [1, 2, 3, 4])
def test_fp32_tiles(gpu_lib, shape, K):
    """The FP32 form's tolerances (test_gpu_fp32.py): species and Phi 2e-4, the
    populations 1e-5 of the largest; the species' totals exact."""
    ek = gpu_lib
    o, s = make_pair(ek, case(shape, K), flags=O.PV, magic=3.0 / 16.0, walls=walls_of(shape), g=(1e-5, 2e-5, -1e-5))
    s.close()
    c = case(shape, K)
    s = ek.EKSystem(shape, nu=c["nu"], rho0=c["rho0"], bjerrum=c["bjerrum"], valence=c["valence"], D=c["D"],
                    bulk=c["bulk"], flags=O.PV | ek.EK_FP32, magic=3.0 / 16.0)
    s.set_field(ek.FIELD_WALL, walls_of(shape).astype(np.float64))
    s.set_field(ek.FIELD_E_EXT, o.E)
    s.set_field(ek.FIELD_BODY_FORCE, o.g)
    perm = perm_to_oracle(ek)
    f = np.empty_like(o.f)
    f[perm] = o.f
    s.set_field(ek.FIELD_POPULATIONS, f.ravel())
    for k in range(K):
        s.set_field(ek.FIELD_SPECIES, o.rho[k].ravel(), component=k)
    before = [s.get_fields(ek.FIELD_SPECIES, k).sum() for k in range(K)]
    o.step(3)
    s.step(3)
    fluid = o.owner == O.FLUID
    for k in range(K):
        got = s.get_fields(ek.FIELD_SPECIES, k)
        assert np.max(np.abs(got - o.rho[k])) <= 2e-4 * np.max(np.abs(o.rho[k]))
        assert got.sum() == before[k]
    assert np.max(np.abs(s.get_fields(ek.FIELD_PHI) - o.phi)) <= 2e-4 * np.max(np.abs(o.phi))
    got = s.get_fields(ek.FIELD_POPULATIONS)[perm]
    assert np.max(np.abs(got - o.f)[:, fluid]) <= 1e-5 * np.max(np.abs(o.f))
