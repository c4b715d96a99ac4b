"""Timed cases of the framework: what a user has it do, over the range of sizes, precisions and options.

Every case is a simulation a user runs: the fields and particles of ``prepare`` stand for a run in
progress (drops, solids and a developed flow), ``run`` advances it by the case's number of time steps and
reads the fields back into device tensors (``pf.Sim.macros``, or the C call ``pf_batch_get_macros_all``
for a batch), or logs the diagnostics on the way (``pf.Sim.run_logged``).

Kinds of cases
  box        one 2D or 3D domain: a drop, fixed solids, periodic or walled in y
  logged     the same, with the FP64 diagnostics every few steps
  particles  one 2D or 3D domain with free particles
  sweep      a batch of uneven 2D domains (drops on a wall, or periodic drops)

Fields come back in the type that the policy carries: float64 (p64), float32 (p32), and the 16-bit
storage type of the populations (fp16, bf16).
"""
import ctypes as C
import math
import random

import numpy as np
import torch

from paper_2311_05097_gb300 import pf

SIXTEEN = ("fp16", "bf16")
DTYPE = {"p64": torch.float64, "p32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}

# bytes of one cell update: every population read and written once, the lagged fields (u, S, phi) read and
# written once, the fixed indicator read once; (16-bit policies: the order parameter's rest population is int64)
CELL_BYTES = {
    2: {"p64": 8 * (36 + 11), "p32": 4 * (36 + 11), "fp16": 4 * 17 + 16 + 44, "bf16": 4 * 17 + 16 + 44},
    3: {"p64": 8 * (52 + 15), "p32": 4 * (52 + 15), "fp16": 4 * 25 + 16 + 60, "bf16": 4 * 25 + 16 + 60},
}
# arithmetic of one cell update that no formulation avoids by much: both collisions in moment space, the
# stencils of phi, mu and the lagged product, the forces and the pressure
CELL_FLOPS = {2: 420.0, 3: 900.0}


def listed():
    return [
        # the Laplace test: the smallest domain that users validate with, in FP64
        dict(name="static_drop_p64", kind="box", dim=2, nx=128, ny=128, precision="p64", solid="none", walls=False,
             phase_model=0, ratio=10.0, tune=False, steps=50),
        # a small box watched closely: ten diagnostics in a hundred steps, ragged sizes
        dict(name="logged_drop_p32", kind="logged", dim=2, nx=250, ny=223, precision="p32", solid="disc", walls=False,
             phase_model=0, ratio=10.0, tune=False, steps=100, every=10),
        # a drop on a cylinder between wall slabs, as a user first runs it (no tuning call)
        dict(name="cylinder_p32", kind="box", dim=2, nx=512, ny=512, precision="p32", solid="cylinder", walls=False,
             phase_model=0, ratio=10.0, tune=False, steps=50),
        # phase separation in a porous medium between bounce-back walls, tuned for a long run
        dict(name="porous_walls_p32", kind="box", dim=2, nx=1024, ny=1024, precision="p32", solid="porous", walls=True,
             phase_model=0, ratio=1.0, tune=True, steps=50),
        # contact-angle sweep: many uneven domains at once, 16-bit storage
        dict(name="sweep_fp16", kind="sweep", count=64, smin=64, smax=512, precision="fp16", walls=False, phase_model=0,
             steps=50),
        # the same kind of sweep in FP64, the reference runs of a study
        dict(name="sweep_p64", kind="sweep", count=16, smin=64, smax=256, precision="p64", walls=False, phase_model=0,
             steps=20),
        # periodic drops with the Allen-Cahn order parameter
        dict(name="sweep_allen_cahn_bf16", kind="sweep", count=40, smin=64, smax=448, precision="bf16", walls=False,
             phase_model=1, steps=50),
        # drainage of a 3D porous medium, the largest domain, 16-bit storage
        dict(name="drainage_3d_fp16", kind="box", dim=3, nx=256, ny=256, nz=256, precision="fp16", solid="porous",
             walls=False, phase_model=0, ratio=10.0, tune=False, steps=24),
        # a 3D box between walls, ragged sizes, FP32
        dict(name="walled_box_3d_p32", kind="box", dim=3, nx=131, ny=100, nz=90, precision="p32", solid="disc", walls=True,
             phase_model=0, ratio=10.0, tune=False, steps=32),
        # one particle falling through an interface in a tall box, 16-bit storage, tuned for a long run
        dict(name="water_entry_fp16", kind="particles", dim=2, nx=1024, ny=2048, precision="fp16", count=1, rmin=40.0,
             rmax=40.0, own=False, walls=False, solid="slab", tune=True, steps=32),
        # mixing by many wetting particles of their own contact angles
        dict(name="mixing_particles_p32", kind="particles", dim=2, nx=512, ny=512, precision="p32", count=16, rmin=20.0,
             rmax=30.0, own=True, walls=False, solid="none", tune=True, steps=32),
        # spheres settling in a 3D box
        dict(name="spheres_3d_p32", kind="particles", dim=3, nx=96, ny=80, nz=112, precision="p32", count=3, rmin=9.0,
             rmax=13.0, own=False, walls=False, solid="none", tune=False, steps=16),
    ]


def draw(rng):
    """One more case of the ranges above; sizes spread over their logarithm, any parity.  (Allen-Cahn runs
    take 16-bit storage: the order parameter's normal jumps where its gradient vanishes, so its last digits
    are those of the rounding at any precision.)"""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["box", "box", "box3", "box3", "logged", "particles", "particles3", "sweep", "sweep"])
    if kind in ("box", "logged"):
        prec = rng.choice(["p64", "p32", "fp16", "bf16"])
        hi = 384 if prec == "p64" else 1024
        c = dict(kind=kind, dim=2, nx=size(48, hi), ny=size(48, hi), precision=prec,
                 solid=rng.choice(["none", "disc", "cylinder", "porous"]), walls=rng.random() < 0.4,
                 phase_model=1 if prec in SIXTEEN and rng.random() < 0.4 else 0, ratio=round(math.exp(rng.uniform(0.0, math.log(10.0))), 3),
                 tune=rng.random() < 0.5, steps=rng.randint(20, 60))
        if c["solid"] == "porous":
            c["ratio"] = 1.0  # phase separation runs at equal densities
        if c["solid"] in ("cylinder", "porous"):
            c["phase_model"] = 0
        if kind == "logged":
            c["every"] = rng.choice([5, 10, 20])
            c["steps"] = c["every"] * rng.randint(3, 8)
        return c
    if kind == "box3":
        prec = rng.choice(["p64", "p32", "fp16", "bf16"])
        hi = 72 if prec == "p64" else 200
        return dict(kind="box", dim=3, nx=size(28, hi), ny=size(28, hi), nz=size(28, hi), precision=prec,
                    solid=rng.choice(["none", "disc", "porous"]), walls=rng.random() < 0.4,
                    phase_model=1 if prec in SIXTEEN and rng.random() < 0.4 else 0, ratio=round(math.exp(rng.uniform(0.0, math.log(10.0))), 3),
                    tune=rng.random() < 0.5, steps=rng.randint(10, 32))
    if kind == "particles":
        return dict(kind="particles", dim=2, nx=size(200, 900), ny=size(200, 900), precision=rng.choice(["p64", "p32", "fp16", "bf16"]),
                    count=rng.randint(1, 16), rmin=14.0, rmax=28.0, own=rng.random() < 0.5, walls=rng.random() < 0.4,
                    solid=rng.choice(["none", "slab"]), tune=rng.random() < 0.5, steps=rng.randint(12, 32))
    if kind == "particles3":
        return dict(kind="particles", dim=3, nx=size(48, 120), ny=size(48, 120), nz=size(48, 120),
                    precision=rng.choice(["p32", "fp16", "bf16"]), count=rng.randint(1, 5), rmin=7.0, rmax=12.0,
                    own=rng.random() < 0.5, walls=rng.random() < 0.4, solid="none", tune=False, steps=rng.randint(8, 16))
    prec = rng.choice(["p64", "p32", "p32", "fp16", "bf16"])
    big = prec != "p64"
    return dict(kind="sweep", count=rng.randint(3, 64 if big else 12), smin=48, smax=size(96, 512 if big else 256),
                precision=prec, walls=rng.random() < 0.3, phase_model=1 if prec in SIXTEEN and rng.random() < 0.4 else 0, steps=rng.randint(20, 50))


# ---- inputs ---------------------------------------------------------------------------------------------

PARAMS = dict(sigma=0.01, D=4.0, M=0.02, eta=0.0, rho1=1.0, rho2=1.0, mu1=0.1, mu2=0.1, d0=0.4, s0=1.0, s1=1.0, s2=1.0,
              s3=1.0, s4=1.0, theta_deg=90.0, Fb=(0.0, 0.0, 0.0), g=(0.0, 0.0, 0.0), solid_eps=1e-3, rep_xi=0.0,
              rep_eps=0.0, wall_circle=(0.0, 0.0, 0.0), phase_model=0)


def _axes(shape):
    """Cell coordinates x, y(, z) as float64 tensors that broadcast over ``shape``."""
    out = []
    for a, n in enumerate(reversed(shape)):
        view = [1] * len(shape)
        view[len(shape) - 1 - a] = n
        out.append(torch.arange(n, device="cuda", dtype=torch.float64).view(view))
    return out


def _dist(shape, centre, walls):
    """Distance of every cell to ``centre`` (minimum image; none across walls in y)."""
    d2 = 0.0
    for a, x in enumerate(_axes(shape)):
        n = shape[len(shape) - 1 - a]
        d = x - centre[a]
        if not (walls and a == 1):
            d = d - n * torch.floor(d / n + 0.5)
        d2 = d2 + d * d
    return torch.sqrt(d2)


def _solid(zeta, D):
    return 0.5 * (1.0 + torch.tanh(2.0 * zeta / D))


def _porous(shape, rng, walls, D):
    """Indicator of discs / spheres of random radii on a jittered grid of spacing about 28 cells."""
    dim = len(shape)
    n = list(reversed(shape))
    cells = [max(1, k // 28) for k in n]
    step = [k / c for k, c in zip(n, cells)]
    zeta = torch.full(shape, -1e9, device="cuda", dtype=torch.float64)
    sites = [(i,) for i in range(cells[0])]
    for a in range(1, dim):
        sites = [s + (i,) for s in sites for i in range(cells[a])]
    for s in sites:
        half = 0.5 * min(step)
        r = rng.uniform(0.55, 0.9) * min(half, 14.0)
        c = [(s[a] + 0.5) * step[a] + rng.uniform(-1.0, 1.0) * max(0.0, half - r - 1.0) for a in range(dim)]
        h = int(r + 6 * D) + 1
        idx, rel = [], []
        for a in range(dim):
            lo = int(math.floor(c[a])) - h
            k = torch.arange(lo, lo + min(2 * h + 2, n[a]), device="cuda")
            if walls and a == 1:
                k = k[(k >= 0) & (k < n[a])]
            idx.append(k % n[a])
            view = [1] * dim
            view[dim - 1 - a] = k.numel()
            rel.append((k.double() - c[a]).view(view))
        d = torch.sqrt(sum(v * v for v in rel))
        at = tuple(k.view([-1 if j == dim - 1 - a else 1 for j in range(dim)]) for a, k in reversed(list(enumerate(idx))))
        zeta[at] = torch.maximum(zeta[at], r - d)
    return _solid(zeta, D)


def _flow(shape, rng, amp, walls):
    """A smooth periodic velocity field of a few Fourier modes (zero at walls in y)."""
    X = _axes(shape)
    n = list(reversed(shape))
    out = []
    for _ in range(len(shape)):
        f = torch.zeros(shape, device="cuda", dtype=torch.float64)
        for _ in range(3):
            ph = rng.uniform(0.0, 2.0 * math.pi)
            arg = ph + sum(2.0 * math.pi * rng.randint(1, 2) * X[a] / n[a] for a in range(len(shape)))
            f += rng.uniform(0.3, 1.0) / 3.0 * torch.sin(arg)
        if walls:
            f = f * torch.sin(math.pi * (X[1] + 0.5) / n[1])
        out.append(amp * f)
    return torch.stack(out)


def _shape(case):
    return (case["ny"], case["nx"]) if case["dim"] == 2 else (case["nz"], case["ny"], case["nx"])


def _box_scene(case, seed):
    """A domain in mid-run: fixed solids, a drop (or noise in a porous medium) and a flow."""
    rng = random.Random(1000003 * seed + 17)
    shape, walls = _shape(case), case["walls"]
    dim, n, D = len(shape), list(reversed(shape)), 4.0
    m = min(n)
    phi0 = torch.zeros(shape, device="cuda", dtype=torch.float64)
    p = dict(PARAMS, phase_model=case["phase_model"], theta_deg=rng.uniform(60.0, 120.0), M=0.05 if dim == 2 else 0.02)
    p.update(rho2=1.0 / case["ratio"], mu2=0.1 * case["ratio"] ** (-2.0 / 3.0), s0=1.6)
    if dim == 3:
        # the D3Q7 rest weight needs d0 <= 1/3; the viscosity cap and s0 of the drainage runs
        p.update(d0=0.3, solid_eps=0.1, s0=1.9, mu2=0.1)
    centre = [n[a] * rng.uniform(0.45, 0.55) for a in range(dim)]
    kind = case["solid"]
    if kind == "disc":
        c = [n[a] * rng.uniform(0.2, 0.26) for a in range(dim)]
        phi0 = _solid(0.15 * m - _dist(shape, c, walls), D)
    elif kind == "cylinder":
        y = _axes(shape)[1]
        y = y + 0.5
        y = (y - n[1] * torch.floor(y / n[1] + 0.5)).abs()
        centre = [n[0] * rng.uniform(0.45, 0.55), n[1] * rng.uniform(0.3, 0.33)]
        phi0 = _solid(8.0 - y, D) + _solid(0.117 * m - _dist(shape, centre, walls), D) * torch.ones(shape, device="cuda", dtype=torch.float64)
        phi0 = phi0.clamp(0.0, 1.0)
        centre = [centre[0], centre[1] + 0.117 * m]
        p.update(sigma=0.001, M=0.1, s0=1.6)
    elif kind == "porous":
        phi0 = _porous(shape, rng, walls, D)
    if kind == "porous" and dim == 2:
        g = torch.Generator(device="cuda").manual_seed(seed + 5)
        noise = torch.rand(shape, device="cuda", dtype=torch.float64, generator=g)
        phi = (1.0 - phi0) * (2.0 * noise - 1.0) * (0.3 if case["phase_model"] else 1.0)
        p.update(sigma=0.001, M=0.1)
    elif kind == "porous":
        x = _axes(shape)[0]
        dx = x - n[0] * rng.uniform(0.1, 0.14)
        dx = dx - n[0] * torch.floor(dx / n[0] + 0.5)
        phi = (1.0 - phi0) * torch.tanh(2.0 * (0.1 * n[0] - dx.abs()) / D)
        p.update(Fb=(1e-6, 0.0, 0.0), theta_deg=rng.uniform(110.0, 130.0))
    else:
        r = m * rng.uniform(0.18, 0.22)
        phi = (1.0 - phi0) * torch.tanh(2.0 * (r - _dist(shape, centre, walls)) / D)
    u = (1.0 - phi0) * _flow(shape, rng, 0.01, walls)
    return dict(shape=shape, phi0=phi0.contiguous(), phi=phi.contiguous(), u=u.contiguous(), params=p, walls=walls, particles=[])


def _particle_scene(case, seed):
    """Free particles around a flat interface (each other's repulsion on when there are several)."""
    rng = random.Random(1000003 * seed + 29)
    shape, walls, dim, D = _shape(case), case["walls"], case["dim"], 4.0
    n = list(reversed(shape))
    phi0 = torch.zeros(shape, device="cuda", dtype=torch.float64)
    X = _axes(shape)
    lo, hi = 0.0, float(n[1])
    if case["solid"] == "slab":
        y = X[1] + 0.5
        phi0 = phi0 + _solid(8.0 - (y - n[1] * torch.floor(y / n[1] + 0.5)).abs(), D)
        lo, hi = 8.0, n[1] - 8.0
    parts = []
    tries = 0
    while len(parts) < case["count"] and tries < 20000:
        tries += 1
        R = rng.uniform(case["rmin"], case["rmax"])
        c = [rng.uniform(0.0, n[a]) for a in range(dim)]
        c[1] = rng.uniform(lo + R + 4.0, hi - R - 4.0) if hi - lo > 2 * R + 9.0 else 0.5 * (lo + hi)
        far = True
        for q in parts:
            d2 = 0.0
            for a in range(dim):
                d = c[a] - q["x"][a]
                d -= n[a] * math.floor(d / n[a] + 0.5)
                d2 += d * d
            far = far and d2 > (R + q["R"] + 4.0) ** 2
        if far:
            parts.append(dict(x=tuple(c) + (0.0,) * (3 - dim), u=(rng.uniform(-5e-3, 5e-3), rng.uniform(-0.02, -0.005), 0.0),
                              w=(0.0, 0.0, rng.uniform(-2e-4, 2e-4)), R=R, rho_p=rng.uniform(1.05, 2.0),
                              theta_deg=rng.uniform(60.0, 120.0) if case["own"] else None))
    solid = phi0.clone()
    u = (1.0 - phi0) * _flow(shape, rng, 0.02, walls)
    for q in parts:
        ind = _solid(q["R"] - _dist(shape, q["x"], walls), D)
        solid = solid + ind
        for a in range(dim):
            u[a] = (1.0 - ind) * u[a] + ind * q["u"][a]
    level = n[1] * rng.uniform(0.42, 0.48)
    phi = (1.0 - solid) * torch.tanh(2.0 * (0.25 * n[1] - (X[1] - 0.5 * level).abs()) / D)
    # equal densities and viscosities, as in the mixing runs: a light particle in a light gas is not stable
    p = dict(PARAMS, sigma=0.001, M=0.1 if dim == 2 else 0.02, theta_deg=rng.uniform(70.0, 110.0), g=(0.0, -1e-6, 0.0), s0=1.6)
    if dim == 3:
        p.update(d0=0.3, solid_eps=0.1, s0=1.9)
    if len(parts) > 1:
        p.update(rep_xi=2.5, rep_eps=1e4)
    return dict(shape=shape, phi0=phi0.contiguous(), phi=phi.contiguous(), u=u.contiguous(), params=p, walls=walls, particles=parts)


def _sweep_sizes(case):
    """Domain sides of a sweep: fixed by the case (the plan), log-uniform and even in x."""
    rng = random.Random(7919 * case["count"] + 31 * case["smin"] + case["smax"])
    out = []
    for _ in range(case["count"]):
        a, b = (math.exp(rng.uniform(math.log(case["smin"]), math.log(case["smax"]))) for _ in range(2))
        out.append((int(b), max(8, int(a) // 2 * 2)))
    return out


def _sweep_scenes(case, seed):
    """Drops on a wall slab (periodic drops for Allen-Cahn), each with its own angle and density ratio."""
    out = []
    for k, shape in enumerate(_sweep_sizes(case)):
        rng = random.Random(1000003 * seed + 101 * k + 3)
        ny, nx = shape
        D, m, walls = 4.0, min(shape), case["walls"]
        phi0 = torch.zeros(shape, device="cuda", dtype=torch.float64)
        ratio = math.exp(rng.uniform(0.0, math.log(20.0)))
        p = dict(PARAMS, M=0.1, rho2=1.0 / ratio, mu2=0.1 * ratio ** (-2.0 / 3.0), s0=1.6, theta_deg=rng.uniform(40.0, 140.0),
                 phase_model=case["phase_model"])
        centre, r = [nx * rng.uniform(0.45, 0.55), ny * rng.uniform(0.45, 0.55)], 0.25 * m
        if not case["phase_model"]:
            y = _axes(shape)[1] + 0.5
            phi0 = phi0 + _solid(8.0 - (y - ny * torch.floor(y / ny + 0.5)).abs(), D)
            centre = [centre[0], 7.5]
        phi = (1.0 - phi0) * torch.tanh(2.0 * (r - _dist(shape, centre, walls)) / D)
        u = (1.0 - phi0) * _flow(shape, rng, 0.005, walls)
        out.append(dict(shape=shape, phi0=phi0.contiguous(), phi=phi.contiguous(), u=u.contiguous(), params=p, walls=walls, particles=[]))
    return out


def _scenes(case, seed):
    if case["kind"] == "sweep":
        return _sweep_scenes(case, seed)
    return [_particle_scene(case, seed) if case["kind"] == "particles" else _box_scene(case, seed)]


# ---- the user's program -----------------------------------------------------------------------------------


def _make_sim(case, sc, stream):
    s = pf.Sim(sc["shape"], precision=case["precision"], stream=stream, walls_y=sc["walls"], **sc["params"])
    for k, q in enumerate(sc["particles"]):
        s.set_particle(k, q["x"], u=q["u"], w=q["w"], R=q["R"], rho_p=q["rho_p"], theta_deg=q["theta_deg"])
    torch.cuda.synchronize()
    s.init(sc["phi0"], sc["phi"], sc["u"])
    return s


def _make_batch(case, scenes, stream):
    b = pf.Batch([s["shape"] for s in scenes], [s["params"] for s in scenes], precision=case["precision"], stream=stream,
                 walls_y=case["walls"])
    torch.cuda.synchronize()
    b.init_all([s["phi0"] for s in scenes], [s["phi"] for s in scenes], [s["u"] for s in scenes])
    return b


_tuned = set()


def prepare(case, seed):
    """A simulation or batch in mid-run on a stream of the caller's, its launch configuration tuned on a scratch
    copy where the case says so (and for every sweep, whose batch then takes the process's cached choice)."""
    scenes = _scenes(case, seed)
    st = torch.cuda.Stream()
    key = repr(sorted((k, v) for k, v in case.items() if k not in ("name", "steps")))
    sweep = case["kind"] == "sweep"
    if key not in _tuned and (sweep or case["tune"]):
        _tuned.add(key)
        if sweep:
            b = _make_batch(case, scenes, st.cuda_stream)
            b.step(256)
            b.close()
        else:
            s = _make_sim(case, scenes[0], st.cuda_stream)
            s.autotune()
            s.close()
    state = dict(kind=case["kind"], stream=st, steps=case["steps"], every=case.get("every", 0), dtype=DTYPE[case["precision"]],
                 shapes=[s["shape"] for s in scenes], np=len(scenes[0]["particles"]))
    if sweep:
        state["batch"] = _make_batch(case, scenes, st.cuda_stream)
    else:
        state["sim"] = _make_sim(case, scenes[0], st.cuda_stream)
        if case["tune"]:
            state["sim"].autotune()  # takes the cached configuration: no steps
    state["out"] = []
    for sc in scenes:
        N, dim = sc["phi"].numel(), len(sc["shape"])
        state["out"].append({k: torch.empty(m * N, device="cuda", dtype=torch.float64) for k, m in (("phi", 1), ("u", dim), ("P", 1))})
    torch.cuda.synchronize()
    return state


def _read(state):
    """The fields of every domain into the program's device tensors."""
    if "sim" in state:
        state["sim"].macros(out=state["out"][0])
        return
    tables = []
    for key in ("phi", "rho", "u", "P", "mu"):
        t = (C.c_void_p * len(state["out"]))(*[o[key].data_ptr() if key in o else None for o in state["out"]])
        tables.append(C.cast(t, C.c_void_p))
    rc = pf.load().pf_batch_get_macros_all(state["batch"]._h, *tables, pf.PF_DEVICE)
    if rc != pf.PF_OK:
        raise pf.PfError(rc, pf.last_error())


def run(state):
    """Advance by the case's steps and read the fields (and the particles, or the logged diagnostics)."""
    with torch.cuda.stream(state["stream"]):
        out = {}
        if state["kind"] == "logged":
            recs = state["sim"].run_logged(state["steps"], state["every"])
            log = torch.tensor([[r["mass"], r["E_F"], r["E_K"]] for r in recs], dtype=torch.float64)
            out["log"] = log if state["dtype"] == torch.float64 else log.float()
        elif "sim" in state:
            state["sim"].step(state["steps"])
        else:
            state["batch"].step(state["steps"])
        _read(state)
        for k in range(state["np"]):
            q = state["sim"].particle(k)
            v = torch.tensor([q["x"], q["u"], q["F"]], dtype=torch.float64)
            out["particle%02d" % k] = v if state["dtype"] == torch.float64 else v.float()
        if "sim" in state:
            shape = state["shapes"][0]
            for key, v in state["out"][0].items():
                out[key] = v.to(state["dtype"]).view((len(shape),) + shape if key == "u" else shape)
        else:
            # one tensor per field, the domains one after another
            for key in ("phi", "u", "P"):
                out[key] = torch.cat([o[key] for o in state["out"]]).to(state["dtype"])
    return out


def work(case):
    """Bytes and operations of one pass: the cell updates of its steps and the fields read back."""
    if case["kind"] == "sweep":
        cells, dim = sum(a * b for a, b in _sweep_sizes(case)), 2
    else:
        dim = case["dim"]
        cells = case["nx"] * case["ny"] * (case["nz"] if dim == 3 else 1)
    size = {"p64": 8, "p32": 4}.get(case["precision"], 2)
    return {"bytes": float(cells) * (case["steps"] * CELL_BYTES[dim][case["precision"]] + (2 + dim) * size),
            "flops": float(cells) * case["steps"] * CELL_FLOPS[dim]}


# ---- the same in plain 64-bit torch -------------------------------------------------------------------------


class _Exact:
    """The scheme of Sec. 3 of arXiv 2311.05097 as full-grid float64 passes."""

    def __init__(self, sc):
        self.shape, self.p, self.walls = sc["shape"], sc["params"], sc["walls"]
        self.dim = d = len(self.shape)
        p = self.p
        self.cs2 = cs2 = p["d0"]
        self.n = list(reversed(self.shape))
        f3 = [(0, 0, 0)]
        for a in range(3):
            for s in (1, -1):
                f3.append(tuple(s if b == a else 0 for b in range(3)))
        e3 = [(sx, sy, 0) for sx in (1, -1) for sy in (1, -1)] + [(sx, 0, sz) for sx in (1, -1) for sz in (1, -1)]
        e3 += [(0, sy, sz) for sy in (1, -1) for sz in (1, -1)]
        w0 = cs2
        if d == 2:
            c = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
            w = [1 - 2 * w0 + w0 * w0] + [(w0 - w0 * w0) / 2] * 4 + [w0 * w0 / 4] * 4
            self.c1, self.w1, self.c2, self.w2 = c, w, c, w
            self.fd = [(v, 1 / 9 if i <= 4 else 1 / 36) for i, v in enumerate(c) if i]
            self.Kc, self.H1, self.H2 = 1 - w0, (1 - 3 * w0) / 2, 2 - 4 * w0
        else:
            self.c1, self.w1 = f3, [1 - 3 * w0] + [w0 / 2] * 6
            self.c2, self.w2 = f3 + e3, [1 - 3 * w0 + 3 * w0 * w0] + [(w0 - 2 * w0 * w0) / 2] * 6 + [w0 * w0 / 4] * 12
            self.fd = [(v, 1 / 18 if i <= 6 else 1 / 36) for i, v in enumerate(self.c2) if i]
            self.Kc, self.H1, self.H2 = 1 - 2 * w0, 1 - 3 * w0, 3 - 7 * w0
        self.MH1, self.MH2 = self._moments(self.c1), self._moments(self.c2)
        self.eta = p["eta"] if p["eta"] > 0 else 2 * p["M"] / cs2
        self.cac = p["phase_model"] == 1
        self.s1phi = 1 / (p["M"] / ((1.0 if self.cac else self.eta) * cs2) + 0.5)
        self.drho, self.rhom = 0.5 * (p["rho1"] - p["rho2"]), 0.5 * (p["rho1"] + p["rho2"])
        self.fixed = sc["phi0"]
        ct = math.cos(math.radians(p["theta_deg"]))
        self.ct = ct
        self.parts = []
        for q in sc["particles"]:
            t = {k: torch.tensor(q[k], device="cuda", dtype=torch.float64) for k in ("x", "u", "w")}
            own = q["theta_deg"] is not None
            t.update(u0=t["u"].clone(), w0=t["w"].clone(), R=q["R"], rho=q["rho_p"], own=own,
                     ct=math.cos(math.radians(q["theta_deg"])) if own else 0.0, F=torch.zeros(3, device="cuda", dtype=torch.float64))
            self.parts.append(t)
        self.own = any(t["own"] for t in self.parts)
        self._indicators()
        phi, u = sc["phi"], sc["u"]
        rho = self.drho * phi + self.rhom
        mu = self._mu(phi)
        S = self._flux(phi, mu, self._grad(phi))
        zero = torch.zeros_like(phi)
        self.f1 = self._feq1(phi, u, mu)
        self.f2 = self._feq2(rho, u, S, zero)
        self.lag = (u, S, phi)

    def _moments(self, c):
        cs2, rows = self.cs2, []
        for v in c:
            x, y, z = (float(t) for t in v)
            hx, hy, hz = x * x - cs2, y * y - cs2, z * z - cs2
            if self.dim == 2:
                rows.append([1, x, y, hx, hy, x * y, x * hy, y * hx, hx * hy])
            elif len(c) == 7:
                rows.append([1, x, y, z, hx, hy, hz])
            else:
                rows.append([1, x, y, z, hx, hy, hz, x * y, x * z, y * z, x * hy, x * hz, y * hx, y * hz, z * hx, z * hy, hx * hy, hx * hz, hy * hz])
        M = torch.tensor(np.array(rows, dtype=np.float64).T.copy(), device="cuda")
        return M, torch.linalg.inv(M)

    def _at(self, a, c, sign=1.0):
        """The field at x + c: periodic, or the mirror image (times ``sign``) beyond a wall in y."""
        for ax, k in enumerate(c[:self.dim]):
            if k == 0:
                continue
            dim = a.dim() - 1 - ax
            if ax == 1 and self.walls:
                ends = [a.narrow(dim, 0, 1) * sign, a, a.narrow(dim, a.shape[dim] - 1, 1) * sign]
                a = torch.cat(ends, dim).narrow(dim, 1 + k, a.shape[dim])
            else:
                a = torch.roll(a, -k, dim)
        return a

    def _grad(self, a, sign=1.0):
        g = [torch.zeros_like(a) for _ in range(self.dim)]
        for c, w in self.fd:
            v = self._at(a, c, sign)
            for k in range(self.dim):
                if c[k]:
                    g[k] += 3.0 * w * c[k] * v
        return torch.stack(g)

    def _lap(self, a):
        out = torch.zeros_like(a)
        for c, w in self.fd:
            out += 6.0 * w * (self._at(a, c) - a)
        return out

    def _rel(self, q):
        r = []
        for a, x in enumerate(_axes(self.shape)):
            d = x - q["x"][a]
            if not (a == 1 and self.walls):
                d = d - self.n[a] * torch.floor(d / self.n[a] + 0.5)
            r.append(d)
        return r

    def _indicators(self):
        D = self.p["D"]
        total, dflt, W, V = self.fixed.clone(), self.fixed.clone(), 0.0, 0.0
        self.ind = []
        for q in self.parts:
            r = self._rel(q)
            k = _solid(q["R"] - torch.sqrt(sum(v * v for v in r)), D)
            self.ind.append((k, r))
            total += k
            if q["own"]:
                W, V = W + q["ct"] * k, V + q["ct"] * k ** 3
            else:
                dflt += k
        self.phi0 = total
        self.W, self.V = self.ct * dflt + W, self.ct * dflt ** 3 + V

    def _mu(self, phi):
        p = self.p
        a, b = 3.0 * p["sigma"] / p["D"], 3.0 * p["D"] * p["sigma"] / 8.0
        p0 = self.phi0
        mu = a * phi * (phi * phi - 1.0) - b * self._lap(phi) + 3.0 * a * p0 * p0 * phi
        if self.own:
            return mu + a * (3.0 * phi * phi * self.W + self.V - self.W) - b * self._lap(self.W)
        return mu + self.ct * (a * p0 * (3.0 * phi * phi + p0 * p0 - 1.0) - b * self._lap(p0))

    def _theta_n(self, phi, g):
        g2 = (g * g).sum(0)
        inv = torch.where(g2 > 1e-24, 1.0 / torch.sqrt(g2.clamp_min(1e-300)), torch.zeros_like(g2))
        return 2.0 / self.p["D"] * (1.0 - phi * phi) * inv * g

    def _flux(self, phi, mu, g):
        grad = g - self._theta_n(phi, g) if self.cac else self._grad(mu)
        return self.p["M"] * self.drho * grad

    def _feq1(self, phi, u, mu):
        em = phi if self.cac else self.eta * mu
        out = []
        for i, (c, w) in enumerate(zip(self.c1, self.w1)):
            cu = sum(c[a] * u[a] for a in range(self.dim))
            out.append(phi + (w - 1.0) * em if i == 0 else w * em + w * cu * phi / self.cs2)
        return torch.stack(out)

    def _feq2(self, rho, u, S, P):
        d, cs2, out = self.dim, self.cs2, []
        T = {(a, b): rho * u[a] * u[b] - 0.5 * (S[a] * u[b] + u[a] * S[b]) for a in range(d) for b in range(a, d)}
        for i, (c, w) in enumerate(zip(self.c2, self.w2)):
            v = (w - 1.0 if i == 0 else w) / cs2 * P
            v = v + w * self._second(c, T)
            v = v + w / cs2 * rho * sum(c[a] * u[a] for a in range(d))
            out.append(v)
        return torch.stack(out)

    def _second(self, c, T):
        d, cs2 = self.dim, self.cs2
        v = sum((c[a] * c[a] - cs2) / (cs2 - cs2 * cs2) * T[a, a] for a in range(d))
        for a in range(d):
            for b in range(a + 1, d):
                if c[a] * c[b]:
                    v = v + c[a] * c[b] / (cs2 * cs2) * T[a, b]
        return v

    def _collide(self, M, f, feq, F, rates):
        """f - Lambda (f - feq) + (1 - Lambda/2) F with Lambda = M^-1 S M."""
        MH, inv = M
        x = f + F
        h = (MH @ (f - feq + 0.5 * F).reshape(len(rates), -1)).view_as(f)
        for k, s in enumerate(rates):
            h[k] *= s
        return x - (inv @ h.reshape(len(rates), -1)).view_as(f)

    def _stream(self, f, c):
        out = torch.empty_like(f)
        for i, v in enumerate(c):
            back = tuple(-k for k in v)
            g = f[i]
            for ax in range(self.dim):
                if v[ax]:
                    g = torch.roll(g, v[ax], g.dim() - 1 - ax)
            out[i] = g
            if self.walls and v[1]:
                # what would come from beyond the wall is the cell's own opposite population
                row = 0 if v[1] > 0 else self.n[1] - 1
                out[i].select(self.dim - 2, row).copy_(f[c.index(back)].select(self.dim - 2, row))
        return out

    def macros(self):
        p, d, cs2 = self.p, self.dim, self.cs2
        phi = self.f1.sum(0)
        rho = self.drho * phi + self.rhom
        g, mu = self._grad(phi), self._mu(phi)
        S = self._flux(phi, mu, g)
        up, Sp, _ = self.lag
        F = mu * g + torch.tensor(p["Fb"][:d], device="cuda", dtype=torch.float64).view([d] + [1] * d)
        for a in range(d):
            for b in range(a + 1, d):
                t = self._grad(Sp[a] * up[b] - up[a] * Sp[b], -1.0 if 1 in (a, b) else 1.0)
                F[b] += 0.5 * t[a]
                F[a] -= 0.5 * t[b]
        if self.parts:
            a3, b3, lap = 3.0 * p["sigma"] / p["D"], 3.0 * p["D"] * p["sigma"] / 8.0, self._lap(phi)
            g0 = self._grad(self.phi0)
            if self.own:
                gW, gV = self._grad(self.W), self._grad(self.V)
                F += 3.0 * a3 * self.phi0 * phi * phi * g0 + (a3 * phi * (phi * phi - 1.0) - b3 * lap) * gW + a3 * phi * gV
            else:
                F += (3.0 * a3 * self.phi0 * phi * phi + self.ct * (a3 * phi * (3.0 * self.phi0 ** 2 + phi * phi - 1.0) - b3 * lap)) * g0
        j = torch.stack([sum(c[a] * self.f2[i] for i, c in enumerate(self.c2) if c[a]) for a in range(d)])
        us = (j + 0.5 * F) / rho
        pen = -self.phi0 * us
        for q, (k, r) in zip(self.parts, self.ind):
            v = self._solid_velocity(q, r)
            for a in range(d):
                pen[a] += k * v[a]
        u = us + 0.5 * pen
        Ft = F + rho * pen
        nu = (0.5 * (p["mu1"] - p["mu2"]) * phi + 0.5 * (p["mu1"] + p["mu2"])) / (rho * (1.0 - self.phi0).clamp_min(p["solid_eps"]))
        i2a, i2b = 0.5 + 2.0 * nu / (1.0 - cs2), 0.5 + nu / cs2
        H = self.Kc * ((1.0 - cs2) / p["s0"] - self.H2 * i2a + self.H1)
        gr = self.drho * g
        ugr = (u * gr).sum(0)
        dt = 2.0 * (u * Ft).sum(0) - ((S * u).sum(0) - (Sp * up).sum(0))
        w0 = self.w2[0]
        P = cs2 / (1.0 - w0) * (self.f2[1:].sum(0) + (0.5 + H) * ugr - w0 * ((rho * u - S) * u).sum(0) / (1.0 - cs2) + 0.5 * self.Kc * dt)
        return dict(phi=phi, rho=rho, mu=mu, S=S, g=g, us=us, u=u, Ft=Ft, i2a=i2a, i2b=i2b, gr=gr, ugr=ugr, P=P)

    def _solid_velocity(self, q, r):
        u, w = q["u"], q["w"]
        if self.dim == 2:
            return [u[0] - w[2] * r[1], u[1] + w[2] * r[0]]
        return [u[0] + w[1] * r[2] - w[2] * r[1], u[1] + w[2] * r[0] - w[0] * r[2], u[2] + w[0] * r[1] - w[1] * r[0]]

    def step(self):
        p, d, cs2 = self.p, self.dim, self.cs2
        m = self.macros()
        up, Sp, php = self.lag
        phi, u, S, rho, Ft, gr, ugr = (m[k] for k in ("phi", "u", "S", "rho", "Ft", "gr", "ugr"))
        force = [self._force(q, k, r, m) for q, (k, r) in zip(self.parts, self.ind)]
        G = phi * u - php * up
        if self.cac:
            G = G + cs2 * self._theta_n(phi, m["g"])
        F1 = torch.stack([w / cs2 * sum(c[a] * G[a] for a in range(d)) if any(c) else torch.zeros_like(phi) for c, w in zip(self.c1, self.w1)])
        s2 = p["s2"]
        r1 = [p["s0"]] + [self.s1phi] * d
        r1 += [s2] * 3 if d == 3 else [s2] * 3 + [p["s3"]] * 2 + [p["s4"]]
        f1 = self._collide(self.MH1, self.f1, self._feq1(phi, u, m["mu"]), F1, r1)
        del F1
        M2 = {}
        for a in range(d):
            for b in range(a, d):
                t = u[a] * Ft[b] + Ft[a] * u[b] - 0.5 * ((S[a] * u[b] + u[a] * S[b]) - (Sp[a] * up[b] + up[a] * Sp[b]))
                t = t + cs2 * (u[a] * gr[b] + gr[a] * u[b])
                M2[a, b] = t + (1.0 - 3.0 * cs2) * ugr if a == b else t
        F2 = torch.stack([w * (ugr + sum(c[a] * Ft[a] for a in range(d)) / cs2 + self._second(c, M2)) for c, w in zip(self.c2, self.w2)])
        s2a, s2b = 1.0 / m["i2a"], 1.0 / m["i2b"]
        if d == 2:
            r2 = [p["s0"]] + [p["s1"]] * 2 + [s2a] * 2 + [s2b] + [p["s3"]] * 2 + [p["s4"]]
        else:
            r2 = [p["s0"]] + [p["s1"]] * 3 + [s2a] * 3 + [s2b] * 3 + [p["s3"]] * 6 + [p["s4"]] * 3
        f2 = self._collide(self.MH2, self.f2, self._feq2(rho, u, S, m["P"]), F2, r2)
        del F2
        self.f1, self.f2 = self._stream(f1, self.c1), self._stream(f2, self.c2)
        self.lag = (u, S, phi)
        if self.parts:
            self._move(force)
            self._indicators()

    def _force(self, q, k, r, m):
        d = self.dim
        v = self._solid_velocity(q, r)
        f = [m["rho"] * k * (v[a] - m["us"][a]) for a in range(d)]
        z = torch.zeros((), device="cuda", dtype=torch.float64)
        F = torch.stack([-f[a].sum() for a in range(d)] + [z] * (3 - d))
        if d == 2:
            T = torch.stack([z, z, -(r[0] * f[1] - r[1] * f[0]).sum()])
        else:
            T = torch.stack([-(r[1] * f[2] - r[2] * f[1]).sum(), -(r[2] * f[0] - r[0] * f[2]).sum(), -(r[0] * f[1] - r[1] * f[0]).sum()])
        return F, T

    def _repulsion(self):
        p, d = self.p, self.dim
        X = [q["x"].cpu().numpy() for q in self.parts]
        out = np.zeros((len(X), 3))
        if not p["rep_eps"] > 0:
            return out

        def size(dist, rr, eps):
            if dist > rr + p["rep_xi"]:
                return 0.0
            return (rr + p["rep_xi"] - dist) ** 2 / eps if dist >= rr else (rr - dist) / eps

        for k, q in enumerate(self.parts):
            if self.walls:
                y = X[k][1]
                low, high = 2.0 * (y + 0.5), 2.0 * (self.n[1] - 0.5 - y)
                best = min(low, high)
                out[k, 1] += size(best, 2.0 * q["R"], 0.5 * p["rep_eps"]) * (low if low <= high else -high)
            for j, o in enumerate(self.parts):
                if j != k:
                    v = np.zeros(3)
                    for a in range(d):
                        v[a] = X[k][a] - X[j][a]
                        if not (a == 1 and self.walls):
                            v[a] -= self.n[a] * math.floor(v[a] / self.n[a] + 0.5)
                    out[k] += size(math.sqrt((v * v).sum()), q["R"] + o["R"], p["rep_eps"]) * v
        return out

    def _move(self, force):
        p, d = self.p, self.dim
        rep = torch.tensor(self._repulsion(), device="cuda")
        g = torch.tensor(p["g"][:d] + (0.0,) * (3 - d), device="cuda", dtype=torch.float64)
        keep = torch.tensor([1.0, 1.0, 0.0 if d == 2 else 1.0], device="cuda", dtype=torch.float64)
        spin = torch.tensor([0.0, 0.0, 1.0] if d == 2 else [1.0] * 3, device="cuda", dtype=torch.float64)
        for k, q in enumerate(self.parts):
            V = math.pi * q["R"] ** 2 if d == 2 else 4.0 / 3.0 * math.pi * q["R"] ** 3
            mass = q["rho"] * V
            I = (0.5 if d == 2 else 0.4) * mass * q["R"] ** 2
            F, T = force[k]
            acc = (F + rep[k] + self.rhom * V * (q["u"] - q["u0"]) + (1.0 - self.rhom / q["rho"]) * mass * g) / mass
            al = (T + I * self.rhom / q["rho"] * (q["w"] - q["w0"])) / I
            q["x"] = q["x"] + q["u"]
            q["u0"], q["w0"] = q["u"], q["w"]
            q["u"], q["w"], q["F"] = q["u"] + keep * acc, q["w"] + spin * al, F

    def diagnostics(self):
        m, p = self.macros(), self.p
        a, b = 3.0 * p["sigma"] / p["D"], 3.0 * p["D"] * p["sigma"] / 8.0
        phi, p0, g = m["phi"], self.phi0, m["g"]
        e = 0.25 * a * (1.0 - phi * phi) ** 2 + 0.5 * b * (g * g).sum(0) + 1.5 * a * p0 * p0 * phi * phi
        e = e + self.ct * (a * p0 * phi * (phi * phi + p0 * p0 - 1.0) + b * (self._grad(p0) * g).sum(0))
        return [phi.sum().item(), e.sum().item(), (0.5 * m["rho"] * (m["u"] ** 2).sum(0)).sum().item()]


def exact(case, seed):
    """What ``run`` returns on a fresh state, from 64-bit full-grid passes in torch."""
    fields, out = [], {}
    for sc in _scenes(case, seed):
        x = _Exact(sc)
        log = []
        for t in range(case["steps"]):
            x.step()
            if case["kind"] == "logged" and (t + 1) % case["every"] == 0:
                log.append(x.diagnostics())
        m = x.macros()
        fields.append({k: m[k] for k in ("phi", "u", "P")})
        if log:
            out["log"] = torch.tensor(log, dtype=torch.float64)
        for k, q in enumerate(x.parts):
            out["particle%02d" % k] = torch.stack([q["x"], q["u"], q["F"]])
        del x, m
    for key in ("phi", "u", "P"):
        out[key] = fields[0][key] if case["kind"] != "sweep" else torch.cat([f[key].reshape(-1) for f in fields])
    return out
