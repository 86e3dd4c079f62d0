"""Fields read into device memory have the bits of the same fields read to the
host: every field of both storage forms, into part of a larger buffer whose other
bytes stay, and to an address no double may be stored to (a copy's work)."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPE = (24, 18, 16)


def box(ek, fp32):
    s = ek.EKSystem(SHAPE, bulk=(1e-3, 2e-3), flags=ek.EK_PV | ek.EK_NEUTRALIZE | (ek.EK_FP32 if fp32 else 0))
    wall = np.zeros(SHAPE[::-1])
    wall[0] = 1.0
    s.set_field(ek.FIELD_WALL_CHARGE, -0.01 * wall)
    s.set_field(ek.FIELD_WALL, wall)
    s.add_particle((12.3, 9.2, 8.6), radius=4.0, charge=-10.0)
    s.set_field(ek.FIELD_E_EXT, np.array([0.004, -0.002, 0.001]))
    s.set_field(ek.FIELD_BODY_FORCE, np.array([1e-5, 0.0, 2e-5]))
    s.step(3)
    return s


def fields(ek):
    return [(ek.FIELD_SPECIES, 0), (ek.FIELD_SPECIES, 1)] + [(f, 0) for f in (
        ek.FIELD_POPULATIONS, ek.FIELD_VELOCITY, ek.FIELD_E_EXT, ek.FIELD_BODY_FORCE, ek.FIELD_WALL,
        ek.FIELD_WALL_CHARGE, ek.FIELD_DENSITY, ek.FIELD_PHI, ek.FIELD_PSI, ek.FIELD_OWNER, ek.FIELD_CHARGE)]


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("before", [0, 7])
def test_into_a_part_of_a_device_tensor(gpu_lib, fp32, before):
    import torch
    ek = gpu_lib
    s = box(ek, fp32)
    for which, comp in fields(ek):
        want = s.get_fields(which, comp).ravel()
        n = want.size
        buf = torch.full((before + n + 5,), 7.25, dtype=torch.float64, device="cuda")
        s.get_fields(which, comp, out=buf[before:before + n])
        got = buf.cpu().numpy()
        assert np.array_equal(got[before:before + n].view(np.uint64), want.view(np.uint64)), (which, comp)
        assert np.all(got[:before] == 7.25) and np.all(got[before + n:] == 7.25), (which, comp)


@pytest.mark.parametrize("fp32", [False, True])
def test_to_an_unaligned_address(gpu_lib, fp32):
    import torch
    ek = gpu_lib
    s = box(ek, fp32)
    for which, comp in fields(ek):
        want = s.get_fields(which, comp).ravel()
        buf = torch.full((8 * want.size + 16,), 0x5a, dtype=torch.uint8, device="cuda")
        s._check(s.lib.ek_get_fields(s.ctx, which, comp, ctypes.c_void_p(buf.data_ptr() + 4), want.size, 1))
        got = buf.cpu().numpy()
        assert got[4:-12].tobytes() == want.tobytes(), (which, comp)
        assert np.all(got[:4] == 0x5a) and np.all(got[-12:] == 0x5a), (which, comp)
