"""Psi on the cells where its column counts can go wrong: centres on the planes
between cells and on those of their 1/16 cubes (an axis neither beyond nor
within a cell but at its edge), a rounding to either side of them, radii whose
surface passes through the cubes' corners, and spheres over the periodic seam,
bit for bit against the octree of the oracle."""
import numpy as np
import pytest

from oracle import ek_oracle as O
from pairs import make_pair

pytestmark = pytest.mark.gpu

CENTRES = {
    "node": (8.0, 8.0, 8.0),
    "corner": (8.5, 8.5, 8.5),
    "edge_lo": (np.nextafter(8.5, 0.0), 8.5, np.nextafter(8.5, 9.0)),
    "float_tie": (8.5 + 2.0 ** -27, 7.5 - 2.0 ** -27, 8.5 - 2.0 ** -50),
    "sixteenth": (8.0625, 8.4375, 7.5625),
    "seam": (0.25, 15.6, 0.5),
    "general": (8.3137, 7.7411, 8.0591),
}


@pytest.mark.parametrize("flags", [0, 16])
@pytest.mark.parametrize("centre", sorted(CENTRES))
def test_psi_bit_for_bit(gpu_lib, centre, flags):
    for R in (1.0, 1.5, 2.5, 3.0, 4.125):
        case = dict(shape=(16, 16, 16), nu=1.0 / 6.0, rho0=1.0, bjerrum=0.7, valence=(1, -1), D=(0.3, 0.3),
                    bulk=(1e-3, 1e-3), E=(0.0, 0.0, 0.0), rho_p=2.0,
                    particles=[dict(pos=CENTRES[centre], radius=R, charge=-5.0)])
        o, s = make_pair(gpu_lib, case, flags=O.PV | flags, perturb=0.0, fixed=True)
        o.step(1)
        s.step(1)
        assert np.array_equal(s.get_fields(gpu_lib.FIELD_PSI), o.psi), R
        s.close()
