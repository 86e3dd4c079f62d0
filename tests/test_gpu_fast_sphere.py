"""A single sphere that moves several cells in one step, in the smallest box it may
have: the box of its old and new cells together is wider than the lattice and holds
nodes twice.  The step ends with an error (the nodes it covers have no fluid
neighbour), but its flags and overlap fractions are those of the new position."""
import numpy as np
import pytest

from oracle import ek_oracle as O

pytestmark = pytest.mark.gpu

KW = dict(nu=1.0 / 6.0, rho0=1.0, bjerrum=0.7, valence=(), D=(), bulk=())


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("vel", [(4.0, 0.0, 0.0), (0.0, -4.0, 0.0), (0.0, 0.0, 4.0), (-5.0, 0.0, 0.0), (0.25, 0.0, 0.0)])
def test_one_step(gpu_lib, fp32, vel):
    ek = gpu_lib
    s = ek.EKSystem((16, 16, 16), flags=ek.EK_PV | (ek.EK_FP32 if fp32 else 0), **KW)
    # heavy: the fluid hardly changes its velocity
    s.add_particle((3.2, 8.1, 7.9), vel=vel, radius=5.0, charge=0.0, rho_p=1e9)
    if max(map(abs, vel)) > 1.0:
        with pytest.raises(ek.EKError) as e:
            s.step(1)
        assert e.value.code == -6
    else:
        s.step(1)
    pos = s.get_particles()[0]["pos"]
    assert np.max(np.abs(pos - (np.array([3.2, 8.1, 7.9]) + vel) % 16.0)) < 1e-6
    o = O.EKOracle(16, 16, 16, flags=O.PV, **KW)
    o.add_particle(tuple(pos), radius=5.0, charge=0.0, rho_p=1.0)
    assert np.array_equal(s.get_fields(ek.FIELD_OWNER), o.owner.astype(np.float64))
    assert np.array_equal(s.get_fields(ek.FIELD_PSI), np.minimum(o.psi, 1.0))
