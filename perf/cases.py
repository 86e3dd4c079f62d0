"""The workloads by which this library's speed is measured: whole calls of its
public entry points (``paper_1607_04572_gb300.ek``) at the sizes, storage forms
and options it is used with.

  step       a box advanced by ``EKSystem.step`` and read back as a program does
             between two stretches of a run: particle records, species, fluid
             velocity, potential (``populations``: the flow's full state too)
  ensemble   independent boxes advanced together by ``EKBatch.step``, read back
  fft        ``poisson_solve``, the periodic Poisson problem by FFT (FP64)
  mg         ``poisson_solve_mg``, the same problem by multigrid (FP64)
  cg         ``poisson_solve_cg``, an inhomogeneous permittivity with
             fixed-potential planes by conjugate gradients (FP64)

What is read from the FP32 storage form is kept by the reading program in
float32, the width the fields are held in.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1607_04572_gb300 import ek

LB = 0.7                      # Bjerrum length
SPECIES = {                   # valences, diffusion coefficients
    2: ((1, -1), (0.3, 0.3)),
    3: ((1, -1, 2), (0.2, 0.3, 0.15)),
}
# box edges the FFT takes (2^a 3^b), the range the boxes are drawn from
EDGES = (24, 32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 324, 384)


def _step(name, shape, fp32, spheres, radius, species=2, salt=1e-3, steps=10, trt=False,
          partial=True, slit=False, populations=False):
    return dict(name=name, kind="step", nx=shape[0], ny=shape[1], nz=shape[2], fp32=fp32,
                spheres=spheres, radius=float(radius), species=species, salt=salt, steps=steps,
                trt=trt, partial=partial, slit=slit, populations=populations)


def _solve(name, kind, shape):
    return dict(name=name, kind=kind, nx=shape[0], ny=shape[1], nz=shape[2])


def listed():
    return [
        # one colloid in the smallest box of a study: launches and latency
        _step("colloid_32", (32, 32, 32), True, 1, 4.0, steps=20),
        # one colloid in the usual box
        _step("colloid_128", (128, 128, 128), True, 1, 8.0, steps=20),
        # a suspension with a divalent counter-ion
        _step("suspension_256", (256, 256, 256), True, 64, 5.0, species=3),
        # the largest box: a suspension of 1000 spheres
        _step("suspension_512", (512, 512, 512), True, 1000, 6.0, salt=5e-4),
        # electro-osmotic flow between charged walls, no particle, ragged box, TRT
        _step("slit_ragged", (192, 108, 72), True, 0, 0.0, trt=True, slit=True, populations=True),
        # the FP64 form: a validation run with the paper's TRT collision
        _step("colloid_64_fp64", (64, 64, 64), False, 1, 4.0, trt=True, populations=True),
        # the FP64 form in the usual box
        _step("colloid_128_fp64", (128, 128, 128), False, 1, 8.0, steps=5),
        # a mobility sweep: independent boxes advanced together
        dict(name="ensemble_64", kind="ensemble", systems=64, steps=20),
        # the standalone solvers: a small ragged box, a large one
        _solve("fft_ragged", "fft", (48, 32, 72)),
        _solve("fft_256", "fft", (256, 256, 256)),
        _solve("mg_128", "mg", (128, 128, 128)),
        _solve("cg_128", "cg", (128, 128, 128)),
    ]


def _draw_shape(rng, lo, hi, edges=EDGES):
    """Edges whose product is spread over the logarithm of [lo, hi]."""
    while True:
        side = math.exp(rng.uniform(math.log(lo), math.log(hi)) / 3.0)
        near = [e for e in edges if 0.6 * side <= e <= 1.6 * side] or [min(edges, key=lambda e: abs(e - side))]
        shape = tuple(rng.choice(near) for _ in range(3))
        if lo <= shape[0] * shape[1] * shape[2] <= hi:
            return shape


def draw(rng):
    what = rng.choice(["step32", "step32", "step32", "step64", "slit", "ensemble", "fft", "mg", "cg"])
    if what in ("step32", "step64"):
        fp32 = what == "step32"
        shape = _draw_shape(rng, 24 ** 3, 384 ** 3 if fp32 else 144 ** 3)
        radius = round(rng.uniform(3.0, min(8.0, (min(shape) - 6) / 2.0)), 2)
        nodes = shape[0] * shape[1] * shape[2]
        most = int(0.02 * nodes / (4.0 / 3.0 * math.pi * radius ** 3))
        spheres = max(1, min(400, int(most * rng.random())))
        case = _step("", shape, fp32, spheres, radius, species=rng.choice([2, 2, 3]) if fp32 else 2,
                     salt=rng.choice([5e-4, 1e-3]), steps=rng.choice([8, 10, 16]), trt=rng.random() < 0.3,
                     partial=rng.random() < 0.8)
    elif what == "slit":
        case = _step("", _draw_shape(rng, 32 ** 3, 216 ** 3), rng.random() < 0.8, 0, 0.0, trt=True,
                     steps=10, slit=True)
        if not case["fp32"]:
            case = dict(case, steps=4)
    elif what == "ensemble":
        case = dict(kind="ensemble", systems=rng.randrange(8, 129), steps=rng.choice([10, 20]))
    elif what == "cg":
        # any edge will do; odd ones cannot be halved and take the diagonal preconditioner
        edges = [e + d for e in (24, 32, 48, 64, 80, 96, 112) for d in ((0, 0, 2, 4, 5) if e < 64 else (0, 2, 4, 8))]
        case = _solve("", "cg", _draw_shape(rng, 24 ** 3, 128 ** 3, edges))
    elif what == "mg":
        case = _solve("", "mg", _draw_shape(rng, 32 ** 3, 192 ** 3))
    else:
        case = _solve("", "fft", _draw_shape(rng, 24 ** 3, 288 ** 3))
    case.pop("name", None)
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _place(rng, shape, count, radius):
    """Random sequential addition of spheres, gaps of at least 4 cells."""
    box = np.array(shape, dtype=np.float64)
    pts = np.empty((0, 3))
    tries = 0
    while len(pts) < count:
        c = rng.random(3) * box
        d = np.abs(pts - c)
        d = np.minimum(d, box - d)
        if not len(pts) or (d * d).sum(axis=1).min() >= (2.0 * radius + 4.0) ** 2:
            pts = np.vstack([pts, c])
        tries += 1
        if tries > 200 * count + 1000:
            break
    return pts


def _setup(case, seed):
    """Plain parameters of a stepped box, from the seed alone."""
    rng = np.random.default_rng(seed)
    shape = (case["nx"], case["ny"], case["nz"])
    z, D = SPECIES[case["species"]]
    R = case["radius"]
    p = dict(shape=shape, nu=1.0 / 6.0, rho0=1.0, bjerrum=LB, valence=z, D=D,
             bulk=(case["salt"],) * len(z), magic=3.0 / 16.0 if case["trt"] else 0.0, rho_p=2.0)
    p["E"] = (rng.uniform(0.003, 0.005), 0.0, rng.uniform(-1e-3, 1e-3))
    p["g"] = (0.0, 0.0, 0.0)
    # surface charges of 0.1 to 0.2 e per cell face (the paper's colloid: 0.15)
    Z = -4.0 * math.pi * R * R * rng.uniform(0.1, 0.2)
    p["particles"] = [(tuple(c), R, Z) for c in _place(rng, shape, case["spheres"], R)]
    if case["slit"]:
        p["g"] = (rng.uniform(0.0, 1e-5), 0.0, 0.0)
        p["wall_charge"] = -rng.uniform(0.005, 0.02)  # per wall node next to the fluid
    return p


def _walls(p):
    """Mask and charge (z, y, x) of a slit: planes z = 0 and z = nz - 1."""
    nx, ny, nz = p["shape"]
    mask = np.zeros((nz, ny, nx))
    mask[0] = mask[-1] = 1.0
    return mask, p["wall_charge"] * mask


def _system(p, flags):
    s = ek.EKSystem(p["shape"], nu=p["nu"], rho0=p["rho0"], bjerrum=p["bjerrum"], valence=p["valence"],
                    D=p["D"], bulk=p["bulk"], flags=flags, magic=p["magic"])
    if "wall_charge" in p:
        mask, charge = _walls(p)
        s.set_field(ek.FIELD_WALL_CHARGE, charge)
        s.set_field(ek.FIELD_WALL, mask)
        s.set_field(ek.FIELD_BODY_FORCE, np.array(p["g"]))
    for pos, radius, charge in p["particles"]:
        s.add_particle(pos, radius=radius, charge=charge, rho_p=p["rho_p"])
    s.set_field(ek.FIELD_E_EXT, np.array(p["E"]))
    return s


def _flags(case):
    return (ek.EK_NEUTRALIZE | (ek.EK_PV if case["partial"] else 0) | (ek.EK_FP32 if case["fp32"] else 0))


def _fields(case):
    """(field, component, values per node) a program reads back."""
    out = [(ek.FIELD_SPECIES, k, 1) for k in range(case["species"])]
    out += [(ek.FIELD_VELOCITY, 0, 3), (ek.FIELD_PHI, 0, 1)]
    return out + ([(ek.FIELD_POPULATIONS, 0, 19)] if case["populations"] else [])


REC_DOUBLES = 19  # an ek_particle record is 19 doubles long: pos, vel, omega, force, torque first


def _records(buf, count, fp32):
    """The particles' state (pos, vel, omega, force, torque) from a buffer of records."""
    rec = np.frombuffer(buf, dtype=np.float64).reshape(-1, REC_DOUBLES)[:count, :15]
    return rec.astype(np.float32 if fp32 else np.float64)


def _ensemble(case, seed):
    """Boxes of a mobility sweep: ragged edges, one sphere each, salt and field
    spread over their logarithms."""
    rng = np.random.default_rng(seed)
    shapes = np.random.default_rng(1607)  # the same boxes for every seed: the buffers keep their sizes
    out = []
    for _ in range(case["systems"]):
        shape = tuple(int(v) for v in shapes.choice([32, 48, 64], 3))
        R = float(shapes.uniform(3.0, 6.0))
        salt = math.exp(rng.uniform(math.log(3e-4), math.log(1e-2)))
        p = dict(shape=shape, nu=1.0 / 6.0, rho0=1.0, bjerrum=LB, valence=(1, -1), D=(0.3, 0.3),
                 bulk=(salt, salt), magic=0.0, rho_p=2.0, g=(0.0, 0.0, 0.0),
                 E=(math.exp(rng.uniform(math.log(2e-3), math.log(1e-2))), 0.0, 0.0))
        pos = tuple(float(v) for v in rng.random(3) * np.array(shape))
        p["particles"] = [(pos, R, -4.0 * math.pi * R * R * float(rng.uniform(0.08, 0.15)))]
        out.append(p)
    return out


def _charge(case, seed):
    """A neutral charge density like a suspension's: smooth ion clouds and noise."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    nz, ny, nx = case["nz"], case["ny"], case["nx"]
    q = 1e-3 * torch.randn(nz, ny, nx, dtype=torch.float64, device="cuda", generator=gen)
    rng = np.random.default_rng(seed)
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") for n in (nz, ny, nx)]
    for _ in range(8):
        width = rng.uniform(2.0, 6.0)
        g = []
        for a, n in zip(ax, (nz, ny, nx)):
            d = (a - rng.random() * n).abs()
            g.append(torch.exp(-0.5 * (torch.minimum(d, n - d) / width) ** 2))
        q += rng.uniform(-0.05, 0.05) * g[0][:, None, None] * g[1][None, :, None] * g[2][None, None, :]
    return q - q.mean()


def _dielectric(case, seed):
    """A low-permittivity sphere in water between electrodes at z = 0 and nz - 1."""
    rng = np.random.default_rng(seed + 1)
    nz, ny, nx = case["nz"], case["ny"], case["nx"]
    z, y, x = torch.meshgrid(*(torch.arange(n, dtype=torch.float64, device="cuda") for n in (nz, ny, nx)),
                             indexing="ij")
    R = 0.16 * min(nx, ny, nz)
    c = [n / 2.0 + rng.uniform(-2.0, 2.0) for n in (nx, ny, nz)]
    r = torch.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2)
    eps = torch.where(r < R, 2.0, 80.0).to(torch.float64)
    fixed = (z == 0) | (z == nz - 1)
    pot = torch.where(z == 0, rng.uniform(0.5, 1.5), -rng.uniform(0.5, 1.5)).to(torch.float64)
    return eps.contiguous(), fixed.to(torch.uint8).contiguous(), pot.contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        s = _system(_setup(case, seed), _flags(case))
        stream = torch.cuda.Stream()
        s.set_stream(stream)
        real = torch.float32 if case["fp32"] else torch.float64
        fields = _fields(case)
        out = [torch.empty(n * s.N, dtype=real, device="cuda") for _, _, n in fields]
        stage = torch.empty(max(n for _, _, n in fields) * s.N, dtype=torch.float64, device="cuda") \
            if case["fp32"] else None
        rec = torch.empty(max(1, s.num_particles()) * REC_DOUBLES * 8, dtype=torch.uint8).pin_memory()
        return dict(case=case, system=s, stream=stream, fields=fields, out=out, stage=stage, rec=rec)
    if kind == "ensemble":
        sys_ = [_system(p, ek.EK_PV | ek.EK_NEUTRALIZE | ek.EK_FP32) for p in _ensemble(case, seed)]
        batch = ek.EKBatch(sys_)
        stream = torch.cuda.Stream()
        batch.set_stream(stream)
        total = sum(s.N for s in sys_)
        out = {k: torch.empty(n * total, dtype=torch.float32, device="cuda") for k, n in (("rho", 2), ("u", 3))}
        stage = torch.empty(5 * total, dtype=torch.float64, device="cuda")
        rec = torch.empty(len(sys_) * REC_DOUBLES * 8, dtype=torch.uint8).pin_memory()
        return dict(case=case, batch=batch, systems=sys_, stream=stream, out=out, stage=stage, rec=rec)
    shape = (case["nx"], case["ny"], case["nz"])
    q = _charge(case, seed)
    st = dict(case=case, shape=shape, q=q, phi=torch.empty_like(q))
    if kind == "fft":
        st["scratch"] = torch.empty(ek.poisson_scratch_bytes(*shape), dtype=torch.uint8, device="cuda")
    elif kind == "mg":
        st["scratch"] = torch.empty(ek.poisson_mg_scratch_bytes(shape), dtype=torch.uint8, device="cuda")
    else:
        st["scratch"] = torch.empty(ek.poisson_cg_scratch_bytes(shape), dtype=torch.uint8, device="cuda")
        st["eps"], st["fixed"], st["pot"] = _dielectric(case, seed)
        st["stream"] = torch.cuda.Stream()
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        s, fp32 = state["system"], case["fp32"]
        s.step(case["steps"])
        n = s.num_particles()
        if n:
            s.get_particles_async(state["rec"])
        with torch.cuda.stream(state["stream"]):
            for (which, comp, _), out in zip(state["fields"], state["out"]):
                if fp32:
                    f64 = state["stage"][:out.numel()]
                    s.get_fields(which, comp, out=f64)
                    out.copy_(f64)
                else:
                    s.get_fields(which, comp, out=out)
        res = {"fields": state["out"]}
        if n:  # the field reads above have waited for the records
            res["particles"] = _records(state["rec"].numpy(), n, fp32)
        return res
    if kind == "ensemble":
        state["batch"].step(case["steps"])
        at = 0
        total = sum(s.N for s in state["systems"])
        rho, u = state["stage"][:2 * total], state["stage"][2 * total:]
        step = REC_DOUBLES * 8
        for i, s in enumerate(state["systems"]):
            s.get_particles_async(state["rec"][i * step:(i + 1) * step])
            for k in range(2):
                s.get_fields(ek.FIELD_SPECIES, k, out=rho[2 * at + k * s.N:2 * at + (k + 1) * s.N])
            s.get_fields(ek.FIELD_VELOCITY, out=u[3 * at:3 * (at + s.N)])
            at += s.N
        state["out"]["rho"].copy_(rho)
        state["out"]["u"].copy_(u)
        return {**state["out"], "particles": _records(state["rec"].numpy(), len(state["systems"]), True)}
    q, phi, shape, scratch = state["q"], state["phi"], state["shape"], state["scratch"]
    if kind == "fft":
        ek.poisson_solve(q, phi, shape, LB, scratch)
    elif kind == "mg":
        ek.poisson_solve_mg(q, phi, shape, LB, scratch)
    else:
        ek.poisson_solve_cg(q, phi, shape, LB, scratch, eps=state["eps"], fixed=state["fixed"],
                            phi_fixed=state["pot"], stream=state["stream"])
    return phi


def work(case):
    """Bytes and operations a pass cannot do without."""
    kind = case["kind"]
    if kind in ("step", "ensemble"):
        if kind == "ensemble":
            shapes = [p["shape"] for p in _ensemble(case, 0)]
            nodes, K, w, read = sum(a * b * c for a, b, c in shapes), 2, 4, 5
        else:
            nodes, K, w = case["nx"] * case["ny"] * case["nz"], case["species"], 4 if case["fp32"] else 8
            read = sum(n for _, _, n in _fields(case))
        # per step: populations and species read and written, the overlap
        # fraction and node class, potential, charge and a spectrum both ways
        per = 2 * 19 * w + 2 * K * w + (w + 1) + 2 * w + 2 * w + 2 * w
        flops = 250 + 18 * (4 + 9 * K) + 7 * 3 * K + 5 * math.log2(nodes)
        return {"bytes": nodes * (case["steps"] * per + 2 * read * w), "flops": nodes * case["steps"] * flops}
    nodes = case["nx"] * case["ny"] * case["nz"]
    if kind == "fft":
        return {"bytes": 16 * nodes, "flops": 5 * nodes * math.log2(nodes)}
    if kind == "mg":  # a dozen V-cycles of four sweeps, residual and transfers
        return {"bytes": 16 * nodes, "flops": 12 * 50 * nodes}
    return {"bytes": 33 * nodes, "flops": 25 * 60 * nodes}


# ---------------------------------------------------------------------------
# the same results in 64 bits by plain torch
# ---------------------------------------------------------------------------
_C = [(0, 0, 0)] + [c for a in range(3) for c in (tuple(int(i == a) for i in range(3)),
                                                  tuple(-int(i == a) for i in range(3)))]
for _a, _b in ((0, 1), (0, 2), (1, 2)):
    for _s in (1, -1):
        _v = [0, 0, 0]
        _v[_a], _v[_b] = 1, _s
        _C += [tuple(_v), tuple(-v for v in _v)]
_W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
_A0 = 1.0 + 2.0 * math.sqrt(2.0)


def _at(a, c):
    """The value at x + c of every node x."""
    return torch.roll(a, (-c[2], -c[1], -c[0]), (-3, -2, -1))


def _poisson64(q):
    lam = [2.0 - 2.0 * torch.cos(2.0 * math.pi * torch.arange(n, dtype=torch.float64, device=q.device) / n)
           for n in q.shape]
    lam = lam[0][:, None, None] + lam[1][None, :, None] + lam[2][None, None, :]
    lam[0, 0, 0] = 1.0
    h = torch.fft.fftn(q) * (4.0 * math.pi * LB) / lam
    h[0, 0, 0] = 0.0
    return torch.fft.ifftn(h).real.contiguous()


class _Sphere:
    def __init__(self, pos, radius, charge, rho_p):
        self.pos, self.R, self.Z = np.array(pos), radius, charge
        self.vel, self.omega, self.force, self.torque, self.trans = (np.zeros(3) for _ in range(5))
        self.mass = rho_p * 4.0 / 3.0 * math.pi * radius ** 3
        self.inertia = 0.4 * self.mass * radius ** 2


class _Box64:
    """The time step of the stepped boxes in 64 bits."""

    def __init__(self, p, partial):
        self.p, self.partial = p, partial
        nx, ny, nz = p["shape"]
        dev = self.dev = torch.device("cuda")
        f64 = dict(dtype=torch.float64, device=dev)
        self.n = (nx, ny, nz)
        self.zv = torch.tensor(p["valence"], **f64)
        self.parts = [_Sphere(np.mod(c, self.n), R, Z, p["rho_p"]) for c, R, Z in p["particles"]]
        self.wall = torch.zeros(nz, ny, nx, dtype=torch.bool, device=dev)
        self.qwall = torch.zeros(nz, ny, nx, **f64)
        if "wall_charge" in p:
            mask, q = _walls(p)
            self.wall, self.qwall = torch.tensor(mask, device=dev) != 0, torch.tensor(q, **f64)
        self._flag()
        fluid = self.owner == -1
        nf = int(fluid.sum())
        bulk = list(p["bulk"])
        net = sum(s.Z for s in self.parts) + float(self.qwall.sum()) + nf * float(np.dot(p["valence"], bulk))
        k = next((k for k, z in enumerate(p["valence"]) if z * net < 0), None)
        if k is not None:
            bulk[k] -= net / (p["valence"][k] * nf)
        self.rho = torch.stack([torch.where(fluid, b, 0.0) for b in torch.tensor(bulk, **f64)])
        self.f = torch.stack([w * p["rho0"] * fluid.to(torch.float64) for w in _W])

    def _flag(self):
        """Owners, overlap fractions (16^3 sub-cubes of a cell: inside 1,
        cut 1/2) and each sphere's cells."""
        nx, ny, nz = self.n
        f64 = dict(dtype=torch.float64, device=self.dev)
        owner = torch.where(self.wall, -2, -1)
        psi = torch.zeros(nz, ny, nx, **f64)
        self.cells = []
        for i, s in enumerate(self.parts):
            lo = [int(math.floor(c - s.R)) - 1 for c in s.pos]
            hi = [int(math.floor(c + s.R)) + 2 for c in s.pos]
            z, y, x = torch.meshgrid(*(torch.arange(lo[a], hi[a], **f64) for a in (2, 1, 0)), indexing="ij")
            x, y, z = x.reshape(-1), y.reshape(-1), z.reshape(-1)
            d = [x - s.pos[0], y - s.pos[1], z - s.pos[2]]
            r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
            flat = (x.long() % nx) + nx * ((y.long() % ny) + ny * (z.long() % nz))
            inside = r2 < s.R * s.R
            part = torch.where(torch.sqrt(r2) < s.R - 0.9, 1.0, 0.0).to(torch.float64)
            cut = torch.nonzero((torch.sqrt(r2) - s.R).abs() <= 0.9).reshape(-1)
            edge = (torch.arange(17, **f64) - 8.0) / 16.0
            for some in cut.split(256):
                lines = [((c[some][:, None] + edge) - o) for c, o in zip((x, y, z), s.pos)]
                sq = [v * v for v in lines]
                corner = (sq[0][:, :, None, None] + sq[1][:, None, :, None] + sq[2][:, None, None, :]) < s.R * s.R
                full = torch.ones(len(some), 16, 16, 16, dtype=torch.bool, device=self.dev)
                for a in (0, 1):
                    for b in (0, 1):
                        for c in (0, 1):
                            full &= corner[:, a:a + 16, b:b + 16, c:c + 16]
                near = [torch.where(v[:, :-1] > 0, sq_[:, :-1], torch.where(v[:, 1:] < 0, sq_[:, 1:], 0.0))
                        for v, sq_ in zip(lines, sq)]
                out = (near[0][:, :, None, None] + near[1][:, None, :, None] + near[2][:, None, None, :]) >= s.R * s.R
                part[some] = (torch.where(full, 1.0, torch.where(out, 0.0, 0.5)).to(torch.float64)
                              .sum(dim=(1, 2, 3)) / 4096.0)
            owner.view(-1)[flat[inside]] = i
            psi.view(-1)[flat] += part
            share = part / part.sum() if self.partial else inside.to(torch.float64) / inside.sum()
            self.cells.append((flat, d, inside, s.Z * share))
        self.owner, self.psi = owner, psi.clamp(max=1.0)

    def _solute(self, fext, E):
        """Force and torque of the solute on each sphere."""
        nx, ny, nz = self.n
        fluid = (self.owner == -1).reshape(-1)
        q = torch.tensordot(self.zv, self.rho, dims=1)
        it = torch.where(fluid.view_as(q), fext - q * torch.tensor(E, dtype=q.dtype, device=self.dev)[:, None, None, None],
                         0.0).reshape(3, -1)
        best = torch.full((nx * ny * nz,), math.inf, dtype=torch.float64, device=self.dev)
        who = torch.full((nx * ny * nz,), -1, dtype=torch.long, device=self.dev)
        regions = []
        for i, s in enumerate(self.parts):
            m = int(math.ceil(s.R)) + 4
            ax = []
            for a, n in enumerate(self.n):
                w = torch.arange(int(math.floor(s.pos[a] - s.R)) - 1 - m, int(math.floor(s.pos[a] + s.R)) + 2 + m,
                                 device=self.dev) % n
                ax.append(torch.unique(w))
            z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
            flat = (x + nx * (y + ny * z)).reshape(-1)
            d = []
            for c, o, n in zip((x, y, z), s.pos, self.n):
                v = c.reshape(-1).to(torch.float64) - o
                v = torch.where(v > 0.5 * n, v - n, v)
                d.append(torch.where(v < -0.5 * n, v + n, v))
            dist = torch.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]) - s.R
            closer = dist < best[flat]
            best[flat[closer]] = dist[closer]
            who[flat[closer]] = i
            regions.append((flat, d))
        F, T, given = [], [], torch.zeros(3, dtype=torch.float64, device=self.dev)
        Et = torch.tensor(E, dtype=torch.float64, device=self.dev)
        cross = lambda d, v: torch.stack([(d[1] * v[2] - d[2] * v[1]).sum(), (d[2] * v[0] - d[0] * v[2]).sum(),
                                          (d[0] * v[1] - d[1] * v[0]).sum()])
        for i, (flat, d) in enumerate(regions):
            mine = (who[flat] == i) & fluid[flat]
            v = torch.where(mine, it[:, flat], 0.0)
            given = given + v.sum(dim=1)
            _, dc, _, qv = self.cells[i]
            F.append(qv.sum() * Et - v.sum(dim=1))
            T.append(cross(dc, Et[:, None] * qv) - cross(d, v))
        rest = (it.sum(dim=1) - given) / len(self.parts)
        return [f - rest for f in F], T

    def step(self):
        p, E, g = self.p, self.p["E"], self.p["g"]
        f64 = dict(dtype=torch.float64, device=self.dev)
        fluid = self.owner == -1
        q = torch.tensordot(self.zv, self.rho, dims=1) + self.qwall
        for flat, _, _, qv in self.cells:
            q.view(-1).index_add_(0, flat, qv)
        self.phi = _poisson64(q)
        # link fluxes and the coupling force
        om = torch.where(fluid, 1.0 - self.psi, 1.0) if self.partial else torch.ones_like(q)
        div, fext = torch.zeros_like(self.rho), torch.zeros(3, *q.shape, **f64)
        for c in _C[1:]:
            link = fluid & _at(fluid, c)
            scale = om * _at(om, c)
            dphi = (self.phi - _at(self.phi, c)) + float(np.dot(E, c))
            for k, (z, D) in enumerate(zip(p["valence"], p["D"])):
                a, b = self.rho[k] / om, _at(self.rho[k], c) / _at(om, c)
                J = torch.where(link, D / (_A0 * math.sqrt(np.dot(c, c))) * ((a - b) + z * 0.5 * (a + b) * dphi) * scale, 0.0)
                div[k] += J
                for d in range(3):
                    if c[d]:
                        fext[d] += (0.5 * c[d] / D) * J
        Fs, Ts = self._solute(fext, E) if self.parts else ([], [])
        # collision
        F = fext + torch.tensor(g, **f64)[:, None, None, None]
        f = torch.where(fluid, self.f, torch.tensor(_W, **f64)[:, None, None, None] * p["rho0"])
        rho = f.sum(dim=0)
        C = torch.tensor(_C, **f64)
        j = torch.tensordot(C.T, f, dims=1)
        u = (j + 0.5 * F) / rho
        tau = 3.0 * p["nu"] + 0.5
        le = -1.0 / tau
        lo = -1.0 / (0.5 + p["magic"] / (tau - 0.5)) if p["magic"] else le
        usq, uF, gg = (u * u).sum(dim=0), (u * F).sum(dim=0), 1.0 + 0.5 * le
        # the velocity of the boundary nodes and their arms
        vb, arm = torch.zeros(3, *q.shape, **f64), torch.zeros(3, *q.shape, **f64)
        for s, (flat, d, inside, _) in zip(self.parts, self.cells):
            w, at = s.omega, flat[inside]
            dd = [v[inside] for v in d]
            v = [s.vel[0] + (w[1] * dd[2] - w[2] * dd[1]), s.vel[1] + (w[2] * dd[0] - w[0] * dd[2]),
                 s.vel[2] + (w[0] * dd[1] - w[1] * dd[0])]
            for a in range(3):
                vb[a].view(-1)[at], arm[a].view(-1)[at] = v[a], dd[a]
        new = torch.zeros_like(f)
        P = len(self.parts)
        Fh, Th = [torch.zeros(3, **f64) for _ in range(P)], [torch.zeros(3, **f64) for _ in range(P)]
        for i, c in enumerate(_C):
            ib = i if i == 0 else (i + 1 if i % 2 else i - 1)
            dot = lambda v: sum((v[a] * c[a] for a in range(3) if c[a]), torch.zeros_like(rho))
            cu, cj, cf = dot(u), dot(j), dot(F)
            plus, minus = 0.5 * (f[i] + f[ib]), 0.5 * (f[i] - f[ib])
            post = (f[i] + le * (plus - _W[i] * rho * (1.0 + 4.5 * cu * cu - 1.5 * usq)) + lo * (minus - 3.0 * _W[i] * cj)
                    + _W[i] * (3.0 * cf + 9.0 * gg * cu * cf - 3.0 * gg * uF))
            if i == 0:
                new[0] = torch.where(fluid, post, 0.0)
                continue
            there = _at(self.owner, c)
            back = tuple(-v for v in c)
            new[i] += _at(torch.where(fluid & (there == -1), post, 0.0), back)
            refl = post - 6.0 * _W[i] * p["rho0"] * dot(torch.stack([_at(v, c) for v in vb]))
            bounce = fluid & (there != -1)
            new[ib] += torch.where(bounce, refl, 0.0)
            for k in range(P):
                m = bounce & (there == k)
                mom = (post + refl)[m]
                if not mom.numel():
                    continue
                dp = [c[a] * mom for a in range(3)]
                ar = [_at(v, c)[m] for v in arm]
                Fh[k] += torch.stack([v.sum() for v in dp])
                Th[k] += torch.stack([(ar[1] * dp[2] - ar[2] * dp[1]).sum(), (ar[2] * dp[0] - ar[0] * dp[2]).sum(),
                                      (ar[0] * dp[1] - ar[1] * dp[0]).sum()])
        u = torch.where(fluid, u, 0.0)
        # volume-of-fluid advection
        au, sg = u.abs(), torch.sign(u)
        adv = torch.zeros_like(self.rho)
        for c in [(a, b, d) for a in (-1, 0, 1) for b in (-1, 0, 1) for d in (-1, 0, 1) if (a, b, d) != (0, 0, 0)]:
            frac = torch.ones_like(q)
            for a in range(3):
                frac = frac * (torch.where(sg[a] == c[a], au[a], 0.0) if c[a] else 1.0 - au[a])
            frac = torch.where(fluid & _at(fluid, c), frac, 0.0)
            for k in range(len(self.rho)):
                amt = self.rho[k] * frac
                adv[k] += _at(amt, tuple(-v for v in c)) - amt
        self.rho, self.f, self.u = self.rho - div + adv, new, u
        for i, s in enumerate(self.parts):
            s.force = (Fh[i] + Fs[i]).cpu().numpy() + s.trans
            s.trans = np.zeros(3)
            s.vel = s.vel + s.force / s.mass
            s.torque = (Th[i] + Ts[i]).cpu().numpy()
            s.omega = s.omega + s.torque / s.inertia
            s.pos = np.mod(s.pos + s.vel, self.n)
        if self.parts:
            old = self.owner
            self._flag()
            self._transitions(old)

    def _transitions(self, old):
        """Fluid and solute of the nodes that a sphere has covered or left."""
        nx, ny, nz = self.n
        new = self.owner
        steady = (old == -1) & (new == -1)
        rho0, f0 = self.rho.clone(), self.f.clone()
        C = np.array(_C, dtype=np.float64)
        for z, y, x in torch.nonzero(old != new).tolist():
            a, b = int(old[z, y, x]), int(new[z, y, x])
            nb = [((z + c[2]) % nz, (y + c[1]) % ny, (x + c[0]) % nx) for c in _C[1:]]
            nb = tuple(torch.tensor(v, device=self.dev) for v in zip(*nb))
            nb = tuple(v[steady[nb]] for v in nb)
            count = len(nb[0])
            if a == -1:  # covered: momentum to the sphere, solute to the neighbours
                self.parts[b].trans += C.T @ f0[:, z, y, x].cpu().numpy()
                self.f[:, z, y, x] = 0.0
                self.rho[:, z, y, x] -= rho0[:, z, y, x]
                for k in range(len(rho0)):
                    self.rho[k][nb] += rho0[k, z, y, x] / count
            else:  # left: equilibrium at the surface's velocity, solute from the neighbours
                s = self.parts[a]
                dens = float(f0.sum(dim=0)[nb].mean()) if count else self.p["rho0"]
                d = np.array([x, y, z]) - s.pos
                d -= np.round(d / self.n) * self.n
                v = s.vel + np.cross(s.omega, d)
                cu = C @ v
                fn = np.array(_W) * dens * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * v @ v)
                self.f[:, z, y, x] = torch.tensor(fn, device=self.dev)
                s.trans -= C.T @ fn
                for k in range(len(rho0)):
                    share = rho0[k][nb] / (count + 1)
                    self.rho[k, z, y, x] += share.sum()
                    self.rho[k][nb] -= share

    def particles(self):
        return np.array([np.concatenate([s.pos, s.vel, s.omega, s.force, s.torque]) for s in self.parts])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fft", "mg"):
        return _poisson64(_charge(case, seed))
    if kind == "cg":
        return _dielectric64(_charge(case, seed), *_dielectric(case, seed))
    if kind == "ensemble":
        rho, u, parts = [], [], []
        for p in _ensemble(case, seed):
            b = _Box64(p, True)
            for _ in range(case["steps"]):
                b.step()
            rho.append(b.rho.reshape(-1))
            u.append(b.u.reshape(-1))
            parts.append(b.particles())
        return {"rho": torch.cat(rho), "u": torch.cat(u),
                "particles": np.concatenate(parts)}
    if case["nx"] * case["ny"] * case["nz"] > 4e6 or case["spheres"] > 8:
        return None  # over 20 seconds
    b = _Box64(_setup(case, seed), case["partial"])
    for _ in range(case["steps"]):
        b.step()
    out = [b.rho[k].reshape(-1) for k in range(case["species"])] + [b.u.reshape(-1), b.phi.reshape(-1)]
    if case["populations"]:  # (those of the nodes inside a sphere mean nothing)
        out.append(None if case["spheres"] else b.f.reshape(-1))
    res = {"fields": out}
    if b.parts:
        res["particles"] = b.particles()
    return res


def _dielectric64(q, eps, fixed, pot):
    """div(eps grad Phi) = -4 pi l_B q with held planes, by plain conjugate
    gradients in 64 bits until the residual stops falling."""
    face = [2.0 * eps * torch.roll(eps, -1, a) / (eps + torch.roll(eps, -1, a)) for a in range(3)]
    free = fixed == 0

    def apply(v):
        out = torch.zeros_like(v)
        for a in range(3):
            flux = face[a] * (v - torch.roll(v, -1, a))
            out += flux - torch.roll(flux, 1, a)
        return out

    diag = sum(f + torch.roll(f, 1, a) for a, f in enumerate(face))
    x = torch.where(free, 0.0, pot)
    r = torch.where(free, 4.0 * math.pi * LB * q - apply(x), 0.0)
    zv = r / diag
    d = zv.clone()
    rz = (r * zv).sum()
    first = float((r * r).sum())
    for it in range(20000):
        Ad = torch.where(free, apply(d), 0.0)
        alpha = rz / (d * Ad).sum()
        x = x + alpha * d
        r = r - alpha * Ad
        zv = r / diag
        new = (r * zv).sum()
        d = zv + (new / rz) * d
        rz = new
        if it % 50 == 49 and float((r * r).sum()) < 1e-30 * first:
            break
    return x
