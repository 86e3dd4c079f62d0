"""The generic line transforms of S1 over the stage radices a plan can take
(FP64 4, 2, 3; FP32 8, 4, 2, 9, 3), edges from the smallest to 1024, few and
many lines, and boxes whose axes mix the specialised and the generic FP32
passes, against the oracle's Poisson solve."""
import numpy as np
import pytest

import workloads
from oracle import ek_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 9, 12), (16, 27, 8), (18, 16, 243), (162, 8, 81), (54, 9, 8),
                                   (1024, 8, 9), (8, 1024, 8), (16, 8, 972), (8, 729, 12), (648, 8, 8),
                                   (72, 72, 54)])
def test_fp64_plans(gpu_lib, shape):
    import torch
    ek = gpu_lib
    nx, ny, nz = shape
    q = np.random.default_rng(21).standard_normal((nz, ny, nx))
    ref = O.poisson(q, 0.7)
    qd = torch.from_numpy(q.ravel()).cuda()
    phi = torch.empty_like(qd)
    spec = torch.empty(ek.poisson_scratch_bytes(nx, ny, nz) // 8, dtype=torch.float64, device="cuda")
    ek.poisson_solve(qd, phi, shape, 0.7, spec)
    got = phi.cpu().numpy().reshape(nz, ny, nx)
    # both sides take the eigenvalues 2 - 2 cos with an absolute error of
    # 2.2e-16, relative to the least of them, (2 pi / n)^2
    lam = (2.0 * np.pi / max(shape)) ** 2
    assert np.max(np.abs(got - ref)) <= max(1e-12, 8 * 2.2e-16 / lam) * np.max(np.abs(ref))


@pytest.mark.parametrize("shape", [(8, 9, 12), (16, 27, 8), (18, 16, 243), (162, 16, 81), (54, 9, 8),
                                   (72, 108, 36), (192, 108, 72), (108, 96, 54), (144, 18, 128), (648, 8, 8)])
def test_fp32_plans(gpu_lib, shape):
    ek = gpu_lib
    nx, ny, nz = shape
    s = ek.EKSystem(shape, nu=1.0 / 6.0, rho0=1.0, bjerrum=0.7, valence=(1, -1), D=(0.3, 0.3),
                    bulk=(1e-3, 1e-3), flags=ek.EK_FP32)
    for k in range(2):
        s.set_field(ek.FIELD_SPECIES, 1e-3 * (1.0 + workloads.perturbation(nx * ny * nz, 0.5, 200 + k)), component=k)
    rho = [s.get_fields(ek.FIELD_SPECIES, k).reshape(nz, ny, nx) for k in range(2)]
    ref = O.poisson(rho[0] - rho[1], 0.7)
    s.run_stage(1)
    got = s.get_fields(ek.FIELD_PHI).reshape(nz, ny, nx)
    # as for the specialised transforms: FP32 rounding of the spectrum
    assert np.max(np.abs(got - ref)) <= 2e-5 * np.max(np.abs(ref))


@pytest.mark.parametrize("shape", [(256, 9, 9), (512, 9, 9), (256, 8, 8), (512, 18, 27), (256, 256, 9), (512, 64, 36),
                                   (256, 36, 512)])
@pytest.mark.parametrize("species", [(1,), (1, -1, 2)])
def test_fp32_row_lines(gpu_lib, shape, species):
    """The x passes of 256 and 512 points (two lines of two rows to a warp, four
    warps to a block): odd and ragged numbers of rows, with a wall charge, one
    and three species."""
    ek = gpu_lib
    nx, ny, nz = shape
    K = len(species)
    s = ek.EKSystem(shape, nu=1.0 / 6.0, rho0=1.0, bjerrum=0.7, valence=species, D=(0.3,) * K,
                    bulk=(1e-3,) * K, flags=ek.EK_FP32)
    q = 1e-3 * workloads.perturbation(nx * ny * nz, 0.5, 301)
    s.set_field(ek.FIELD_WALL_CHARGE, q)
    q = q.reshape(nz, ny, nx)
    for k in range(K):
        s.set_field(ek.FIELD_SPECIES, 1e-3 * (1.0 + workloads.perturbation(nx * ny * nz, 0.5, 302 + k)), component=k)
        q = q + species[k] * s.get_fields(ek.FIELD_SPECIES, k).reshape(nz, ny, nx)
    ref = O.poisson(q, 0.7)
    s.run_stage(1)
    got = s.get_fields(ek.FIELD_PHI).reshape(nz, ny, nx)
    # as above: FP32 rounding of the spectrum
    assert np.max(np.abs(got - ref)) <= 2e-5 * np.max(np.abs(ref))
    s.close()
