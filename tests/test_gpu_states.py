"""The FP32 form's states, bit for bit.  Its float sums round by their order, and a
change of 1e-8 in a particle's motion can carry a level-4 cube of a Psi over the
sphere's surface a step earlier or later, which shows in the velocities next to it
(1e-3 of their rms).  So the order is fixed: the states after some steps are the
recorded ones, and neither the segments of S2 nor the batch change a bit of them."""
import hashlib

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

# SHA-256 (first 16 hex digits) of species, populations and velocity after 20 steps
# on GB300, CUDA 13.0
RECORDED = {
    "box 0": "1c7957ea5b89863f",
    "box 1": "70d384220f2fdc16",
    "box 2": "ea20818cc7c3ce82",
    "box 3": "2001f8b2baff13a0",
    "box 4": "ac6be4b6e3179885",
    "box 5": "e732215224fc1825",
    "several": "e3d4720e5b7718fa",
    "slit": "cf52ef2661e6c94d",
}


def make(ek, w, magic=0.0):
    s = ek.EKSystem(w["shape"], nu=w["nu"], rho0=w["rho0"], bjerrum=w["bjerrum"], valence=w["valence"], D=w["D"],
                    bulk=w["bulk"], flags=ek.EK_PV | ek.EK_NEUTRALIZE | ek.EK_FP32, magic=magic)
    if "walls" in w:
        s.set_field(ek.FIELD_WALL_CHARGE, -0.01 * w["walls"])
        s.set_field(ek.FIELD_WALL, w["walls"])
    for p in w["particles"]:
        s.add_particle(p["pos"], radius=p["radius"], charge=p["charge"], rho_p=w["rho_p"])
    s.set_field(ek.FIELD_E_EXT, np.array(w["E"], dtype=np.float64))
    return s


def fields(ek, s, K):
    out = [s.get_fields(ek.FIELD_SPECIES, k) for k in range(K)]
    return [np.asarray(v, dtype=np.float64).ravel() + 0.0 for v in  # (-0 as 0)
            out + [s.get_fields(ek.FIELD_POPULATIONS), s.get_fields(ek.FIELD_VELOCITY)]]


def digest(ek, s, K):
    h = hashlib.sha256()
    for v in fields(ek, s, K):
        h.update(v.tobytes())
    return h.hexdigest()[:16]


def several():
    """Three species, TRT, spheres close to one another, over the seam."""
    return dict(shape=(64, 48, 24), nu=1.0 / 6.0, rho0=1.0, bjerrum=0.7, valence=(1, -1, 2), D=(0.2, 0.3, 0.15),
                bulk=(1e-3,) * 3, E=(0.004, -0.002, 0.001), rho_p=2.0,
                particles=[dict(pos=c, radius=R, charge=-40.0)
                           for c, R in (((0.3, 0.2, 23.7), 4.0), ((20.1, 24.4, 12.2), 5.0), ((45.7, 30.2, 3.1), 3.5))])


def slit():
    walls = np.zeros((48, 32, 96))
    walls[0] = walls[-1] = 1.0
    return dict(shape=(96, 32, 48), nu=1.0 / 6.0, rho0=1.0, bjerrum=0.7, valence=(1, -1), D=(0.3, 0.3),
                bulk=(1e-3, 1e-3), E=(0.003, 0.0, 0.0), particles=[], rho_p=2.0, walls=walls)


def test_an_ensemble_ends_in_the_recorded_states(gpu_lib):
    ek = gpu_lib
    ws = workloads.batch_ensemble(6, seed=2024)
    sys_ = [make(ek, w) for w in ws]
    b = ek.EKBatch(sys_)
    b.step(20)
    assert {"box %d" % i: digest(ek, s, 2) for i, s in enumerate(sys_)} == \
        {k: v for k, v in RECORDED.items() if k.startswith("box")}


def test_boxes_stepped_alone_end_in_the_recorded_states(gpu_lib):
    ek = gpu_lib
    got = {}
    for i, w in enumerate(workloads.batch_ensemble(6, seed=2024)):
        s = make(ek, w)
        s.step(20)
        got["box %d" % i] = digest(ek, s, 2)
    for name, w, K in (("several", several(), 3), ("slit", slit(), 2)):
        s = make(ek, w, magic=3.0 / 16.0)
        s.step(20)
        got[name] = digest(ek, s, K)
    assert got == RECORDED


# flat and ragged boxes: plane groups of three and of four planes, and of both
SHAPES = [(32, 16, 18), (24, 36, 27), (64, 16, 32), (36, 24, 16)]


@pytest.mark.parametrize("fused", [0, 1])
def test_the_segments_of_s2_do_not_change_a_step(gpu_lib, fused):
    ek = gpu_lib

    def boxes():
        out = []
        for n in SHAPES:
            w = dict(several(), shape=n, particles=[dict(pos=(n[0] - 0.4, 0.7 * n[1], 0.3), radius=4.0, charge=-20.0)])
            out.append(make(ek, w))
        return out

    alone = boxes()
    for s in alone:
        s.step(7)
    for planes in (1, 2, 3, 4, 5, 8, 16, 64):
        sys_ = boxes()
        b = ek.EKBatch(sys_)
        b.set_config(planes_per_block=planes, fused=fused)
        b.step(7)
        for s, t in zip(sys_, alone):
            for u, v in zip(fields(ek, s, 3), fields(ek, t, 3)):
                assert np.array_equal(u, v), (planes, s.shape)
            for key in ("pos", "vel", "omega", "force"):
                assert np.array_equal(s.get_particles()[0][key], t.get_particles()[0][key]), (planes, key)
        b.close()
        for s in sys_:
            s.close()


@pytest.mark.parametrize("fp64_too", [False, True])
def test_a_batch_starts_from_a_configuration_the_tuner_tries(gpu_lib, fp64_too):
    """Its segment length is one of the tuner's, in both forms, and the tuner also
    tries the configuration in use: it cannot leave the batch slower."""
    ek = gpu_lib
    ws = workloads.batch_ensemble(3, seed=2025, edges=(32,))
    sys_ = [make(ek, w) for w in ws]
    if fp64_too:  # no fused form
        w = ws[0]
        sys_.append(ek.EKSystem(w["shape"], valence=w["valence"], D=w["D"], bulk=w["bulk"], flags=ek.EK_PV))
    b = ek.EKBatch(sys_)
    assert b.config()["fused"] == (0 if fp64_too else 1)
    assert b.config()["planes_per_block"] == 2  # 12 tile columns: the shortest it tries
    b.set_config(planes_per_block=5)
    cfg, _ = b.tune(2)
    assert cfg["planes_per_block"] in (2, 4, 5, 8)
    b.close()
