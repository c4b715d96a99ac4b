"""Kernels at the sizes where their work splits can go wrong (edges of pieces,
tiles and chunks, remainders, the smallest grids), against the FP64 oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_05097_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf():
    from paper_2311_05097_gb300 import build
    build.build()
    from paper_2311_05097_gb300 import pf as _pf
    _pf.load()
    return _pf


def _pair(pf, c, steps, precision="p64", particles=(), walls=False, config=None):
    g = pf.Sim(c["shape"], precision=precision, walls_y=walls, **c["params"])
    o = O.OracleSim(c["shape"], O.make_params(**c["params"]))
    if walls:
        o.set_walls(True)
    for k, q in enumerate(particles):
        g.set_particle(k, **q)
        o.set_particle(k, O.Particle(**q))
    g.init(c["phi0"], c["phi"], c.get("u"))
    o.init(c["phi0"], c["phi"], c.get("u"))
    if config is not None:
        g.set_config(*config)
    g.step(steps)
    o.step(steps)
    return g, o


@pytest.mark.parametrize("shape,walls", [
    ((4, 4), False), ((5, 31), True), ((33, 32), False), ((37, 65), True), ((700, 33), False),
    ((4, 4, 4), False), ((5, 6, 33), True), ((9, 8, 64), False),
])
def test_diagnostics_row_pieces(pf, shape, walls):
    """The diagnostics' row pieces of 32 cells: rows shorter than, equal to and
    one past a piece, more rows than warps.  Sums of FP64 terms in another
    order: 1e-12 relative, as the fields' parity."""
    c = W.small_case(shape, seed=3, solid=min(shape) > 8, theta_deg=70.0, u_amp=0.01)
    g, o = _pair(pf, c, 3, walls=walls)
    for _ in range(2):  # (the ticket of the last block is reset by each call)
        dg, do = g.diagnostics(), o.diagnostics()
        for k in ("mass", "E_F", "E_K"):
            assert abs(dg[k] - do[k]) <= 1e-12 * max(abs(do[k]), 1e-3), (k, dg[k], do[k])
        assert dg["nan_flag"] == 0


@pytest.mark.parametrize("precision,tol", [("p32", dict(phi=5e-6, u=2e-4, P=2e-4)), ("fp16", dict(phi=1e-4, u=2e-2, P=2e-2))])
@pytest.mark.parametrize("shape,walls,unit,model", [
    ((4, 4, 4), False, True, 0), ((5, 9, 33), False, True, 0), ((5, 9, 33), True, True, 0), ((33, 8, 31), False, False, 0),
    ((7, 17, 65), True, False, 0), ((67, 7, 32), False, True, 0), ((9, 10, 35), True, False, 1),
])
def test_pair_3d_chunk_edges(pf, precision, tol, shape, walls, unit, model):
    """The 3D two-cells step: chunks of one plane and of unequal length, an empty
    second chunk, tiles past the domain's end in x and y, walls on the tile's
    first and last row, general rates and the Allen-Cahn lattice.  Bounds: ten
    steps of a few FP32 roundings (6e-8) on fields of size 1 (phi), 0.01 (u) and
    the flow populations' 2^-11 rounding in the 16-bit policy."""
    if model and precision == "fp16":
        pytest.skip("Allen-Cahn movers carry phi itself: the bound above is for Cahn-Hilliard ones")
    c = W.small_case(shape, seed=11, solid=min(shape) > 6, theta_deg=75.0, u_amp=0.01, rho_ratio=2.0, mu_ratio=2.0)
    c["params"].update(phase_model=model, solid_eps=0.1)
    if not unit:
        c["params"].update(s0=1.3, s1=0.9, s2=1.1, s3=1.2, s4=0.8, eta=0.0 if model else 0.3)
    g, o = _pair(pf, c, 10, precision=precision, walls=walls)
    gm, om = g.macros(), o.macros()
    for k, t in tol.items():
        assert np.abs(gm[k] - om[k]).max() <= t * max(np.abs(om[k]).max(), 1e-3), k
    if precision == "fp16":
        assert abs(g.diagnostics()["mass"] - c["phi"].sum()) <= 1e-12 * np.abs(c["phi"]).sum()


def test_pair_3d_batch_equals_single_runs(pf):
    """A batch of 3D domains (descriptors from the device table) and single runs
    (descriptor as a kernel parameter) compute the same bits up to the packed
    arithmetic's contraction: FP32 rounding over ten steps."""
    cases = [W.small_case(s, seed=k, solid=True, theta_deg=60.0, u_amp=0.01, rho_ratio=2.0) for k, s in
             enumerate([(9, 12, 33), (20, 8, 16), (13, 13, 13)])]
    b = pf.Batch([c["shape"] for c in cases], [c["params"] for c in cases], precision="p32")
    b.init_all([c["phi0"] for c in cases], [c["phi"] for c in cases], [c["u"] for c in cases])
    b.step(10)
    for i, c in enumerate(cases):
        s = pf.Sim(c["shape"], precision="p32", **c["params"])
        s.init(c["phi0"], c["phi"], c["u"])
        s.step(10)
        x, y = b.macros(i), s.macros()
        for k in ("phi", "u"):
            assert np.abs(x[k] - y[k]).max() <= 5e-6 * max(np.abs(y[k]).max(), 1e-3), k


# boxes wide enough for one image per tile (reach R + 10 D in FP64, R + 5 D in FP32 arithmetic), and
# too small for it; particles across periodic faces, beside walls, of their own angle
@pytest.mark.parametrize("precision,shape,walls", [
    ("p64", (130, 20, 134), False), ("p64", (12, 17, 37), True), ("p32", (92, 96, 100), False), ("p32", (30, 92, 95), True),
    ("fp16", (92, 23, 96), False), ("p32", (11, 9, 33), False),
])
def test_moving_3d_near_lists(pf, precision, shape, walls):
    """The 3D particle step's lists of near particles: FP64 at 1e-12; the FP32 and
    16-bit policies within a few roundings of four steps (FP32 6e-8, 16-bit
    movers 2^-11 of sizes below 0.02), forces relative to the largest one."""
    nz, ny, nx = shape
    c = W.small_case(shape, seed=4, solid=False, u_amp=0.005, rho_ratio=1.0, mu_ratio=1.0)
    R = min(4.0, 0.2 * min(shape))
    # (no cell exactly half a box from a centre: its minimum image is not unique)
    parts = [dict(x=(0.4, 0.5 * ny + 0.31, 0.6 * nz + 0.07), u=(0.01, 0.002, -0.004), w=(0.001, 0.0, 0.002), R=R, rho_p=2.0),
             dict(x=(0.55 * nx + 0.03, 0.3 * ny + 0.11, nz - 0.7), u=(0.0, 0.01, 0.0), R=0.8 * R, rho_p=1.5, theta_deg=60.0),
             dict(x=(nx - 5.2, ny - (R + 1.5 if walls else 0.2), 0.25 * nz + 0.09), u=(0.0, 0.0, 0.01), R=R, rho_p=1.2)]
    for q in parts:
        c["phi"] = (1.0 - W.disc(shape, q["x"], q["R"], 4.0)) * c["phi"]
    g, o = _pair(pf, c, 4, precision=precision, particles=parts, walls=walls)
    gm, om = g.macros(), o.macros()
    tol = dict(p64=(1e-12, 1e-12, 1e-12), p32=(2e-6, 1e-4, 1e-4), fp16=(1e-4, 2e-2, 2e-2))[precision]
    for k, t in zip(("phi", "u", "P"), tol):
        assert np.abs(gm[k] - om[k]).max() <= t * max(np.abs(om[k]).max(), 1e-3), k
    F = max(np.abs(np.array(o.particle(k).F)).max() for k in range(3))
    for k in range(3):
        pg, po = g.particle(k), o.particle(k)
        assert np.abs(np.array(pg["x"]) - np.array(po.x)).max() <= 1e-6 * max(shape), k
        assert np.abs(np.array(pg["F"]) - np.array(po.F)).max() <= (1e-11 if precision == "p64" else 2e-3) * F, k


# 16 x 8 half tiles (few cells) and 32 x 8 tiles (one per SM), ragged in both directions; solid-free
# frames, frames at a solid's rim, walls; unit rates (s0 free) and general ones
@pytest.mark.parametrize("shape,walls,solid,unit", [
    ((128, 128), False, False, True), ((7, 33), False, False, True), ((9, 17), True, True, True),
    ((61, 50), False, True, True), ((151, 250), False, True, True), ((40, 47), True, True, False),
])
def test_fp64_2d_unit_and_half_tiles(pf, shape, walls, solid, unit):
    """The FP64 2D step (unit-rate collisions, shared divisions, half tiles): the oracle at 1e-12."""
    c = W.small_case(shape, seed=8, solid=solid, theta_deg=65.0, u_amp=0.01, rho_ratio=3.0, mu_ratio=2.0)
    c["params"].update(s0=1.6, solid_eps=1e-3)
    if not unit:
        c["params"].update(s1=0.9, s2=1.1, s3=1.2, s4=0.8, eta=0.3)
    g, o = _pair(pf, c, 6, precision="p64", walls=walls)
    gm, om = g.macros(), o.macros()
    for k in ("phi", "u", "P", "mu"):
        assert np.abs(gm[k] - om[k]).max() <= 1e-12 * max(np.abs(om[k]).max(), 1e-3), k


@pytest.mark.parametrize("shapes,precision,walls", [
    ([(7, 9), (33, 40), (64, 70)], "p64", True), ([(50, 36), (8, 130)], "fp16", False), ([(5, 6, 33), (40, 9, 8)], "p32", True),
])
def test_device_outputs_equal_host_ones(pf, shapes, precision, walls):
    """Fields written by the pass into the caller's device arrays, arrays that it may not write (overlapping
    ones: copies), fields left out, and the host's copies: the same bits."""
    import ctypes as C
    import torch
    cases = [W.small_case(s, seed=k, solid=min(s) > 6, u_amp=0.01) for k, s in enumerate(shapes)]
    b = pf.Batch(shapes, [c["params"] for c in cases], precision=precision, walls_y=walls)
    b.init_all([c["phi0"] for c in cases], [c["phi"] for c in cases], [c["u"] for c in cases])
    b.step(3)
    host = b.macros_all()
    dim, keys = len(shapes[0]), ("phi", "rho", "u", "P", "mu")
    for left_out, shared in ((None, False), ("rho", False), (None, True)):
        bufs, tables = [], []
        for s in shapes:
            N = int(np.prod(s))
            one = torch.full(((4 + dim) * N + 1,), float("nan"), dtype=torch.float64, device="cuda")
            at, o = 1, {}
            for k in keys:
                o[k] = one[at:at + (dim if k == "u" else 1) * N]
                at += 0 if shared and k == "phi" else o[k].numel()  # (shared: rho over phi)
            bufs.append(o)
        for k in keys:
            t = (C.c_void_p * len(shapes))(*[None if k == left_out else o[k].data_ptr() for o in bufs])
            tables.append(C.cast(t, C.c_void_p))
        assert pf.load().pf_batch_get_macros_all(b._h, *tables, pf.PF_DEVICE) == pf.PF_OK
        for i, o in enumerate(bufs):
            for k in keys:
                got = o[k].cpu().numpy()
                if k == left_out:
                    assert np.isnan(got).all()
                elif not (shared and k == "phi"):
                    assert np.array_equal(got, np.asarray(host[i][k]).reshape(-1)), (i, k)


@pytest.mark.parametrize("shape", [(4, 5), (17, 33), (16, 64), (47, 95)])
@pytest.mark.parametrize("precision", ["p32", "fp16", "bf16"])
@pytest.mark.parametrize("unit", [True, False])
def test_pair_2d_unit_rates(pf, shape, precision, unit):
    """The tiled two-cells step at unit and general rates, tiles ragged in both directions, against the oracle:
    a few roundings of six steps (FP32 6e-8; 16-bit movers 2^-11 and 2^-8 of sizes below 0.02)."""
    tol = dict(p32=dict(phi=2e-6, u=1e-4), fp16=dict(phi=1e-4, u=2e-2), bf16=dict(phi=1e-3, u=0.2))[precision]
    c = W.small_case(shape, seed=5, solid=min(shape) > 8, theta_deg=75.0, u_amp=0.01, rho_ratio=2.0, mu_ratio=2.0)
    c["params"].update(solid_eps=0.1)
    if not unit:
        c["params"].update(s0=1.3, s1=0.9, s2=1.1, s3=1.2, s4=0.8, eta=0.3)
    for cfg in ((32, 16, 1, 0), (64, 8, 1, 0)):
        g, o = _pair(pf, c, 6, precision=precision, config=cfg)
        gm, om = g.macros(), o.macros()
        for k, t in tol.items():
            assert np.abs(gm[k] - om[k]).max() <= t * max(np.abs(om[k]).max(), 1e-3), (cfg, k)


@pytest.mark.parametrize("shapes", [[(5, 8), (9, 10)], [(61, 72), (257, 130), (8, 66)]])
def test_tuned_strip_segments(pf, shapes):
    """Batches whose domains are shorter than the shortest segment and longer than the longest: every candidate
    the tuner runs computes the same update."""
    cases = [W.small_case(s, seed=k, solid=False, u_amp=0.01) for k, s in enumerate(shapes)]
    b = pf.Batch(shapes, [c["params"] for c in cases], precision="p32")
    b.init_all([c["phi0"] for c in cases], [c["phi"] for c in cases], [c["u"] for c in cases])
    b.step(256)
    for i, c in enumerate(cases):
        s = pf.Sim(c["shape"], precision="p32", **c["params"])
        s.init(c["phi0"], c["phi"], c["u"])
        s.step(256)
        x, y = b.macros(i), s.macros()
        # FP32 roundings of 256 steps (random: 6e-8 sqrt(256) of phi, 16 times that as the fields' bound)
        assert np.abs(x["phi"] - y["phi"]).max() <= 2e-5, i


@pytest.mark.parametrize("d0", [0.4, 0.3, 1.0 / 3.0])
def test_unit_rates_keep_momentum_fp32(pf, d0):
    """A uniform flow without an interface keeps its velocity: the FP32 step's weights of a moment's axis and
    diagonal shares add up exactly, so only roundings remain (6e-8 a step, as a random walk over 200 steps; a
    drift of 3e-8 a step would reach 6e-6)."""
    c = W.small_case((20, 36), seed=1, solid=False, rho_ratio=1.0, mu_ratio=1.0)
    c["params"].update(d0=d0, s0=1.6)
    u = np.zeros((2, 20, 36))
    u[0], u[1] = 0.013, -0.007
    g = pf.Sim(c["shape"], precision="p32", **c["params"])
    g.init(c["phi0"], np.ones(c["shape"]), u)
    g.set_config(32, 8, 0, 0)
    g.step(200)
    m = g.macros()
    for a in range(2):
        assert abs(m["u"][a].mean() / u[a, 0, 0] - 1.0) <= 6e-8 * np.sqrt(200.0) * 2.0


# boxes narrower than the tile (32 x 8 in FP32 arithmetic, 16 x 8 in FP64) in x and y, down to the smallest:
# frame cells lie several box lengths from a particle's nearest image
@pytest.mark.parametrize("precision,shape,walls", [
    ("p32", (9, 7, 4), False), ("p32", (5, 4, 8), False), ("p32", (7, 9, 11), True), ("p32", (10, 5, 16), False),
    ("p32", (4, 6, 17), True), ("fp16", (8, 5, 6), False), ("fp16", (6, 9, 15), True),
    ("p64", (8, 9, 5), False), ("p64", (4, 5, 6), False), ("p64", (9, 4, 9), False), ("p64", (6, 7, 7), True),
    ("p64", (4, 4, 4), False),
])
def test_moving_3d_narrow_boxes(pf, precision, shape, walls):
    """The minimum image of the 3D particle step in boxes of less than a tile: FP64 at 1e-12; FP32 and the
    16-bit policy within a few roundings of four steps (6e-8; movers 2^-11 of sizes below 0.02)."""
    nz, ny, nx = shape
    c = W.small_case(shape, seed=9, solid=False, u_amp=0.005, rho_ratio=1.0, mu_ratio=1.0, D=2.0)
    c["params"].update(solid_eps=0.1)
    R = min(2.0, 0.25 * min(shape))
    # (no cell exactly half a box from a centre: its minimum image is not unique)
    parts = [dict(x=(0.46 * nx + 0.03, 0.5 * ny + 0.31, 0.6 * nz + 0.07), u=(0.01, 0.002, -0.004), w=(0.001, 0.0, 0.002),
                  R=R, rho_p=2.0),
             dict(x=(0.9 * nx + 0.01, 0.3 * ny + 0.11, nz - 0.7), u=(0.0, 0.01, 0.0), R=0.8 * R, rho_p=1.5, theta_deg=60.0)]
    for q in parts:
        c["phi"] = (1.0 - W.disc(shape, q["x"], q["R"], 2.0)) * c["phi"]
    g, o = _pair(pf, c, 4, precision=precision, particles=parts, walls=walls)
    gm, om = g.macros(), o.macros()
    tol = dict(p64=(1e-12, 1e-12, 1e-12), p32=(2e-6, 1e-4, 1e-4), fp16=(1e-4, 2e-2, 2e-2))[precision]
    for k, t in zip(("phi", "u", "P"), tol):
        assert np.abs(gm[k] - om[k]).max() <= t * max(np.abs(om[k]).max(), 1e-3), k
    F = max(np.abs(np.array(o.particle(k).F)).max() for k in range(2))
    for k in range(2):
        pg, po = g.particle(k), o.particle(k)
        assert np.abs(np.array(pg["x"]) - np.array(po.x)).max() <= 1e-6 * max(shape), k
        assert np.abs(np.array(pg["F"]) - np.array(po.F)).max() <= (1e-11 if precision == "p64" else 2e-3) * F, k


def test_moving_3d_simulations_on_several_threads(pf):
    """Host threads launch the same 3D kernels with different numbers of particles: the dynamic shared memory that
    the larger ones need stays allowed whatever the others launch in between."""
    import threading

    def sim(count):
        c = W.small_case((12, 14, 40), seed=2, solid=False)
        s = pf.Sim(c["shape"], precision="p32", **c["params"])
        for k in range(count):
            s.set_particle(k, x=(4.0 + 0.65 * k, 5.0 + 0.1 * k, 6.0), R=1.5, rho_p=1.5, theta_deg=60.0)
        s.init(c["phi0"], c["phi"])
        s.step(2)
        return s

    failed = []

    def work(s, n):
        try:
            for _ in range(n):
                s.diagnostics()
        except pf.PfError as e:
            failed.append(str(e))

    threads = [threading.Thread(target=work, args=(sim(count), 4000)) for count in (1, 1, 1, 50, 50)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed


@pytest.mark.parametrize("shape,count", [((64, 72), 12), ((40, 40, 44), 6)])
@pytest.mark.parametrize("precision", ["p64", "fp16"])
def test_repulsion_in_one_call_equals_single_steps(pf, shape, count, precision):
    """Particles that push one another, every step's launches following on at once (one call of many steps) and
    each step waited for: the same bits."""
    c = W.small_case(shape, seed=3, solid=False, rho_ratio=1.0, mu_ratio=1.0)
    c["params"].update(rep_xi=2.5, rep_eps=1e4, solid_eps=0.1)
    n = list(reversed(shape))
    parts = []
    for k in range(count):
        i = np.array([k % 3, k // 3 % 4, k % 2])[:len(n)]
        parts.append(dict(x=[float(v) for v in 14.2 * i + 9.1], u=[0.002 * (-1) ** k] + [0.0] * (len(n) - 1), R=6.0, rho_p=3.0))
        c["phi"] = (1.0 - W.disc(shape, parts[-1]["x"], 6.0, 4.0)) * c["phi"]
    sims = []
    for _ in range(2):
        s = pf.Sim(shape, precision=precision, **c["params"])
        for k, q in enumerate(parts):
            s.set_particle(k, **q)
        s.init(c["phi0"], c["phi"])
        s.set_config(16 if len(n) == 3 and precision == "p64" else 32, 8, 0, 0)
        sims.append(s)
    sims[0].step(48)
    for _ in range(48):
        sims[1].step(1)
        sims[1].sync()
    for k in range(count):
        a, b = sims[0].particle(k), sims[1].particle(k)
        assert all(a[f] == b[f] for f in ("x", "u", "w", "F", "T")), k
        assert a["x"][0] != parts[k]["x"][0]
    assert np.array_equal(sims[0].macros()["phi"], sims[1].macros()["phi"])


@pytest.mark.parametrize("where", ["direct", "overlapping", "host"])
def test_timed_out_step_leaves_outputs_alone(pf, monkeypatch, where):
    """A readback after a step whose bounded wait ran out returns the error and writes nothing into the caller's
    arrays: those the pass writes itself, those it copies to, one domain and a whole batch."""
    import ctypes as C
    import torch
    shapes = [(32, 64), (40, 96)]
    cases = [W.small_case(s, seed=1, solid=False) for s in shapes]
    for batch in (False, True):
        monkeypatch.setenv("PF_WAIT_POLLS", "1")
        if batch:
            g = pf.Batch(shapes, [c["params"] for c in cases], precision="fp16")
        else:
            g = pf.Sim(shapes[0], precision="fp16", **cases[0]["params"])
        monkeypatch.delenv("PF_WAIT_POLLS")
        if batch:
            g.init_all([c["phi0"] for c in cases], [c["phi"] for c in cases])
        else:
            g.init(cases[0]["phi0"], cases[0]["phi"])
        g.set_config(64, 128, 4)
        g.step(1)
        bufs = [torch.full((6 * s[0] * s[1],), 7.0, dtype=torch.float64, device="cpu" if where == "host" else "cuda")
                for s in shapes]
        N = [s[0] * s[1] for s in shapes]
        ptrs = []
        for k in range(5):  # phi, rho, u, P, mu (overlapping: rho over phi)
            at = {"overlapping": [0, 0, 2, 4, 5]}.get(where, [0, 1, 2, 4, 5])[k]
            ptrs.append([b.data_ptr() + 8 * at * n for b, n in zip(bufs, N)])
        w = pf.PF_HOST if where == "host" else pf.PF_DEVICE
        if batch:
            tables = [C.cast((C.c_void_p * 2)(*p), C.c_void_p) for p in ptrs]
            rc = pf.load().pf_batch_get_macros_all(g._h, *tables, w)
        else:
            rc = pf.load().pf_get_macros(g._h, *[C.c_void_p(p[0]) for p in ptrs], w)
        assert rc == pf.PF_ETIMEOUT
        assert all(bool((b == 7.0).all()) for b in bufs)


@pytest.mark.parametrize("shape,R", [((12, 10, 500), 200.0), ((112, 104, 128), 40.0)])
def test_moving_3d_indicator_rounding_fp32(pf, shape, R):
    """The particle's indicator in FP32 arithmetic: the squared distance of the FP64 offsets, rounded once (in a
    box too small for one image, and in one wide enough).  At phi = 1 and 90 degrees mu_phi = c_pen phi0^2; the
    bound is tanhf's and phi's roundings (2 ulp of 6e-8 each, the latter through c_dw and c_pen).  Distances in
    FP32 throughout would differ by an ulp of R, 4e-6 and 1.5e-5."""
    D, sigma = 1.0, 0.01
    nz, ny, nx = shape
    c = W.small_case(shape, seed=1, solid=False, D=D, theta_deg=90.0)
    x = (0.5 * nx + 0.337, 0.5 * ny + 0.171, 0.5 * nz - 0.219)
    g = pf.Sim(shape, precision="p32", **c["params"])
    g.set_particle(0, x=x, R=R, rho_p=1.0)
    g.init(np.zeros(shape), np.ones(shape))
    mu = g.macros()["mu"] / (9.0 * sigma / D)
    d = [np.arange(n) - v for n, v in zip((nx, ny, nz), x)]
    dx, dy, dz = (v - n * np.rint(v / n) for v, n in zip(d, (nx, ny, nz)))
    r2 = dx[None, None, :] ** 2 + dy[None, :, None] ** 2 + dz[:, None, None] ** 2
    f = np.float32
    z = f(2.0) * (f(R) - np.sqrt(r2.astype(f))) / f(D)
    p0 = 0.5 * (1.0 + np.tanh(z.astype(np.float64)))
    assert np.abs(mu - p0 * p0).max() <= 1e-6


def _finish(nx, ny, seg, places=304, band=4):
    """When the last of a domain's strip items ends, in rows, handed out longest first to the chip's places."""
    import heapq
    strips = (nx + 63) // 64
    rows = [seg] * (strips * (ny // seg)) + [ny % seg] * (strips if ny % seg else 0)
    load = [0] * places
    for r in rows:
        heapq.heapreplace(load, load[0] + (r + band - 1) // band * band + 10)
    return max(load)


def test_strip_segment_of_other_sizes(pf):
    """The segment length tuned on one domain is not taken over by another size of the same cell-count class:
    that one's items end within a tenth of the earliest, as the tuned ones do (56 rows of 692 x 761: 1.74)."""
    for shape in ((1024, 1024), (761, 692), (940, 1100), (600, 1000)):
        c = W.small_case(shape, seed=1, solid=False)
        s = pf.Sim(shape, precision="p32", walls_y=True, **c["params"])
        s.init(c["phi0"], np.ones(shape))
        s.autotune()
        tx, seg, _, kernel = s.config()
        if kernel != 4:
            continue
        ny, nx = shape
        best = min(_finish(nx, ny, k) for k in range(8, 260, 4))
        assert _finish(nx, ny, seg) <= 1.1 * best, (shape, seg)


# 32 x 8 tiles: 64 (one per SM or fewer), 300 (two), 352 (three: not overlapped), 512 (four), 640 (two waves)
@pytest.mark.parametrize("ny", [64, 300, 352, 512, 640])
@pytest.mark.parametrize("precision,walls", [("p32", False), ("fp16", False), ("fp16", True), ("p64", True)])
def test_overlapped_steps_equal_waited_ones(pf, ny, precision, walls):
    """The single-cell step launched over the step before it, where the rule says so, and steps waited for one by
    one: the same bits."""
    shape = (ny, 250)
    c = W.small_case(shape, seed=2, solid=True, u_amp=0.01, rho_ratio=2.0, mu_ratio=2.0)
    sims = []
    for _ in range(2):
        s = pf.Sim(shape, precision=precision, walls_y=walls, **c["params"])
        s.init(c["phi0"], c["phi"], c["u"])
        sims.append(s)
    sims[0].step(20)
    for _ in range(20):
        sims[1].step(1)
        sims[1].sync()
    a, b = sims[0].macros(), sims[1].macros()
    assert all(np.array_equal(a[k], b[k]) for k in a)


@pytest.mark.parametrize("precision", ["p32", "fp16", "bf16"])
@pytest.mark.parametrize("config", [(64, 12, 4, 0), (64, 20, 4, 0), (64, 60, 4, 0), (64, 61, 4, 0), (64, 100, 4, 0),
                                    (32, 16, 1, 0), (64, 8, 1, 0)])
def test_two_cells_steps_against_single_cell(pf, precision, config):
    """Strip segments that leave one row, fit the domain and exceed it, and the tiled two-cells step, against the
    single-cell step of the same policy at unit rates: six steps of FP32 roundings, which flip a stored 16-bit
    population now and then (an ulp, 2^-10 and 2^-7, of populations near 0.005 in phi and 0.001 in the flow, a few
    per cell and step: of u's 0.01 less than 0.2% and 2%)."""
    tol = dict(p32=(2e-6, 1e-4), fp16=(6e-5, 2.5e-3), bf16=(5e-4, 2e-2))[precision]
    c = W.small_case((61, 72), seed=6, solid=True, theta_deg=75.0, u_amp=0.01, rho_ratio=2.0, mu_ratio=2.0)
    c["params"].update(solid_eps=0.1)
    out = []
    for cfg in ((32, 8, 0, 0), config):
        s = pf.Sim(c["shape"], precision=precision, **c["params"])
        s.init(c["phi0"], c["phi"], c["u"])
        s.set_config(*cfg)
        s.step(6)
        out.append(s.macros())
    a, b = out
    assert np.abs(a["phi"] - b["phi"]).max() <= tol[0]
    for k in ("u", "P"):
        assert np.abs(a[k] - b[k]).max() <= tol[1] * np.abs(a[k]).max(), k
