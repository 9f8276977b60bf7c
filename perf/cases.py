"""Workloads a user of the library has it do, for timing and comparing builds.

Every case is a dict of plain values.  ``prepare`` builds what a user's program
holds before the call (a simulation in the middle of its stage and a checkpoint
of it in device memory, a batch of runs, an adjoint run's buffers), ``run`` is
one pass through the public entry points, ``work`` the bytes and operations a
pass cannot do without and ``exact`` the same results in 64 bits from plain
torch, where the inputs are given explicitly.

A stepping pass restarts from the checkpoint, advances some steps and reads
the fields back, as a program that scans, retries or optimises does; so every
pass does the same work, wherever the passes before it stopped.
"""
import math

import numpy as np
import torch

import paper_1011_0917_gb300 as P
from paper_1011_0917_gb300 import workloads as W

EB, CUR = 0x3F, 0x1C0  # component masks: E and B; J


# ------------------------------------------------------------------ the cases


def _boost2d(**kw):
    """The 100 MeV stage of the paper in 2D (gamma 13): every boosted 2D run."""
    c = dict(kind="stage", dim=2, nx=256, ny=1, nz=8192, dx=1.0, dz=1 / 32, gamma=13.0, order=1, passes=2, fp64=False,
             explicit=False, ne=0.001, a0=1.0, waist=20.0, fwhm=10.0, slots=8.0, window=False, snapshots=0,
             advance=500, steps=20)
    c.update(kw)
    return c


def _boost3d(**kw):
    """The same stage in 3D, the plasma filling the box."""
    c = _boost2d(dim=3, nx=128, ny=128, nz=256, slots=10.0, advance=120, steps=10)
    c.update(kw)
    return c


def _loaded(**kw):
    """A thermal plasma and fields that the user brings along (host particles)."""
    c = dict(kind="loaded", dim=2, nx=64, ny=1, nz=256, gamma=1.0, order=2, passes=1, fp64=True, n=60000, ions=0,
             steps=4)
    c.update(kw)
    return c


def _adjoint(**kw):
    c = dict(kind="adjoint", dim=2, nx=128, ny=1, nz=1536, gamma=5.0, order=1, passes=2, profile=8, steps=100, every=25)
    c.update(kw)
    return c


def listed():
    return [
        # the lab-frame 2D stage: the smallest grid in use, a step is a few short launches
        dict(_boost2d(nx=64, nz=512, dx=0.5, dz=1 / 16, gamma=1.0, passes=1, ne=0.01, waist=8.0, fwhm=5.0,
                      advance=256, steps=16), name="lab2d_64x512"),
        # the boosted 2D stage at full length, mid-run
        dict(_boost2d(), name="boost2d_256x8192"),
        # the high-boost stage: quadratic shape, 4 filter passes, records relative to the drift
        dict(_boost2d(nx=512, nz=2048, gamma=130.0, order=2, passes=4, ne=5.7e-5, a0=1.5, waist=50.0, fwhm=30.0,
                      advance=400, steps=8), name="boost2d_g130_quad_512x2048"),
        # gamma 5 in a moving window with lab-frame snapshots taken on the way
        dict(_boost2d(nx=256, nz=1000, gamma=5.0, passes=1, ne=0.004, a0=2.0, waist=16.0, fwhm=4.0, window=True,
                      snapshots=8, advance=600, steps=20), name="window2d_snapshots_256x1000"),
        # the debug precision, on a thermal plasma handed over by the user
        dict(_loaded(), name="thermal2d_fp64_quad_64x256"),
        # 3D with sides that no tile divides, particles handed over by the user
        dict(_loaded(dim=3, nx=75, ny=52, nz=99, order=1, fp64=False, n=900000, steps=3), name="thermal3d_75x52x99"),
        # the boosted 3D stage on a slab (parameter studies, profiles)
        dict(_boost3d(), name="boost3d_128x128x256"),
        # the throughput workload, as large as fits a card three times over
        dict(_boost3d(nx=256, ny=256, nz=512, advance=150, steps=6), name="boost3d_256x256x512"),
        # reading results: the lab-frame view, the charge density and the sums
        dict(_loaded(dim=3, nx=96, ny=80, nz=160, gamma=13.0, order=1, fp64=False, n=600000, ions=400000, steps=0),
             kind="view", name="view3d_96x80x160"),
        # a scan over stage parameters: uneven runs stepped together
        dict(kind="batch", runs=16, nx=128, nz_lo=1024, nz_hi=4096, advance=200, steps=80, name="batch16_c4"),
        # gradients of a run with respect to its profile and laser
        dict(_adjoint(), name="adjoint2d_128x1536"),
        dict(_adjoint(dim=3, nx=48, ny=48, nz=128, gamma=13.0, profile=0, steps=40, every=10),
             name="adjoint3d_48x48x128"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lab2d", "boost2d", "boost2d", "quad2d", "window2d", "boost3d", "boost3d", "loaded2d",
                       "loaded3d", "view", "batch", "adjoint2d", "adjoint3d"])
    if kind == "lab2d":
        nz = _log(rng, 200, 2000)
        return _boost2d(nx=_log(rng, 24, 300), nz=nz, dx=0.5, dz=1 / 16, gamma=1.0, passes=rng.choice([0, 1, 2]),
                        ne=0.01, waist=8.0, fwhm=5.0, order=rng.choice([1, 1, 2]), advance=min(nz // 2, 400),
                        steps=rng.randint(10, 24))
    if kind == "boost2d":
        nz = _log(rng, 300, 8000)
        return _boost2d(nx=_log(rng, 40, 260), nz=nz, gamma=rng.choice([5.0, 13.0, 30.0]),
                        passes=rng.choice([1, 2, 2, 3]), explicit=rng.choice([False, False, True]),
                        a0=round(rng.uniform(0.5, 2.0), 3), advance=min(nz // 4, 500), steps=rng.randint(10, 20))
    if kind == "quad2d":
        return _boost2d(nx=_log(rng, 64, 512), nz=_log(rng, 300, 2000), gamma=rng.choice([13.0, 130.0]), order=2,
                        passes=4, ne=5.7e-5, a0=1.5, waist=50.0, fwhm=30.0, advance=rng.randint(100, 400),
                        steps=rng.randint(4, 8))
    if kind == "window2d":
        nz = _log(rng, 300, 1000)
        return _boost2d(nx=_log(rng, 48, 256), nz=nz, gamma=5.0, passes=1, ne=0.004, a0=2.0, waist=16.0, fwhm=4.0,
                        window=True, snapshots=rng.randint(2, 16), advance=int(0.6 * nz), steps=rng.randint(10, 24))
    if kind == "boost3d":
        nz = _log(rng, 60, 400)
        return _boost3d(nx=_log(rng, 40, 160), ny=_log(rng, 40, 160), nz=nz, passes=rng.choice([1, 2, 2, 4]),
                        explicit=rng.choice([False, False, True]), advance=min(nz // 2, 150), steps=rng.randint(4, 10))
    if kind == "loaded2d":
        nx, nz = _log(rng, 24, 200), _log(rng, 100, 600)
        return _loaded(nx=nx, nz=nz, order=rng.choice([1, 2]), fp64=rng.choice([False, True]),
                       passes=rng.choice([0, 1, 2, 5]), n=rng.randint(2, 8) * nx * nz // 2, steps=rng.randint(1, 5))
    if kind == "loaded3d":
        return _loaded(dim=3, nx=rng.randint(20, 80), ny=rng.randint(20, 80), nz=rng.randint(40, 100),
                       order=rng.choice([1, 1, 2]), fp64=rng.choice([False, False, True]),
                       passes=rng.choice([1, 2]), n=_log(rng, 100000, 500000), steps=rng.randint(1, 3))
    if kind == "view":
        return dict(_loaded(dim=3, nx=rng.randint(30, 100), ny=rng.randint(30, 100), nz=rng.randint(60, 200),
                            gamma=rng.choice([5.0, 13.0, 30.0]), order=rng.choice([1, 2]), fp64=False,
                            n=_log(rng, 100000, 600000), ions=_log(rng, 50000, 400000), steps=0), kind="view")
    if kind == "batch":
        return dict(kind="batch", runs=rng.randint(4, 20), nx=rng.choice([64, 96, 128, 150]),
                    nz_lo=rng.randint(300, 1000), nz_hi=rng.randint(1200, 3000), advance=rng.randint(100, 200),
                    steps=20 * rng.randint(2, 4))
    if kind == "adjoint2d":
        steps = rng.randint(40, 120)
        return _adjoint(nx=rng.randint(40, 150), nz=_log(rng, 300, 1500), gamma=rng.choice([5.0, 13.0]),
                        order=rng.choice([1, 1, 2]), profile=rng.randint(1, 8), steps=steps,
                        every=rng.randint(10, steps))
    return _adjoint(dim=3, nx=rng.randint(20, 48), ny=rng.randint(20, 48), nz=rng.randint(40, 120), gamma=13.0,
                    profile=rng.choice([0, 2]), steps=rng.randint(20, 40), every=rng.randint(8, 20))


# ------------------------------------------------------------- what a user has


def _sim(c, seed, stream=None, slots=None):
    return P.Simulation(dim=c["dim"], nx=c["nx"], ny=c["ny"], nz=c["nz"], dx=c.get("dx", 1.0), dy=1.0,
                        dz=c.get("dz", 1 / 32), gamma_boost=c["gamma"], shape_order=c["order"],
                        filter_passes=c["passes"], precision=P.PIC_FP64 if c.get("fp64") else P.PIC_FP32,
                        seed=W.SEED0 + 7919 * seed, slots_per_cell=slots or c["slots"],
                        explicit_ions=c.get("explicit", False), stream=stream)


def _checkpoint(sim):
    n = P.pic_state_bytes(sim.ctx)
    buf = torch.empty(n, dtype=torch.uint8, device="cuda")
    P.pic_get_state(sim.ctx, buf.data_ptr(), n, True)
    return buf


def _restore(sim, buf):
    P.pic_set_state(sim.ctx, buf.data_ptr(), buf.numel(), True)


def _read(sim, mask, out, frame=P.PIC_FRAME_BOOST):
    P.pic_get_fields(sim.ctx, mask, frame, out.data_ptr(), out.numel() * out.element_size(), True)
    return out


def _fields_out(sim, n):
    return torch.empty((n,) + sim.shape3, dtype=sim.dtype, device="cuda")


def prepare(case, seed):
    return {"stage": _prepare_stage, "loaded": _prepare_loaded, "view": _prepare_loaded, "batch": _prepare_batch,
            "adjoint": _prepare_adjoint}[case["kind"]](case, seed)


def _ppc(c):
    return (2, 2 if c["dim"] == 3 else 1, 2)


def _prepare_stage(c, seed):
    rng = np.random.default_rng(seed)
    a0 = c["a0"] * float(rng.uniform(0.9, 1.1))
    sim = _sim(c, seed)
    hz = sim.sizes.hz
    if c["window"]:  # it follows once the pulse is well inside
        sim.set_moving_window(0.74, 0.4 * c["nz"] * hz, 16)
    if c["gamma"] == 1.0:
        sim.load_plasma(c["ne"], 4.0, max(0.9 * c["nz"] * hz, 8.0), 2.0, _ppc(c), 0.1)
        sim.launch_laser(a0, c["waist"], c["fwhm"], t_peak=6.0)
    else:  # the plasma starts a few cells ahead of the antenna and streams in for the whole run
        z0 = c["gamma"] * 10 * hz
        sim.load_plasma(c["ne"], z0, z0 + 1e6, 2.0, _ppc(c), 0.1)
        sim.launch_laser(a0, c["waist"], c["fwhm"], t_peak=0.5)
    sim.step(c["advance"])
    s = {"case": c, "sim": sim, "eb": _fields_out(sim, 6), "cur": _fields_out(sim, 3)}
    if c["snapshots"]:
        # the events of snapshot j lie at simulation time t' = T_j / gamma - beta z'
        d = sim.diagnostics()
        g, b = c["gamma"], sim.sizes.beta
        lz = c["nz"] * hz
        T = [g * (d.t + b * (d.z_window + f * lz)) for f in (0.05, 0.45)]
        n = c["snapshots"]
        z_lo, z_hi = b * T[0] + d.z_window / g, b * T[1] + (d.z_window + lz) / g
        sim.btd_setup(n, T[0], (T[1] - T[0]) / max(1, n - 1), z_lo, (z_hi - z_lo) / 2000, 2000, 1)
        s["snap"] = [torch.empty(6 * 2000 * c["nx"] + 2000, dtype=torch.float32, device="cuda") for _ in range(n)]
    s["state"] = _checkpoint(sim)
    return s


def _bring(c, seed):
    """The fields and particles of the "loaded" and "view" cases, in 64 bits:
    positions on a lattice of 2^-20 cells and momenta that 32 bits hold."""
    rng = np.random.default_rng(1000003 * (seed % 65521) + 17)
    shape = (c["nz"] + 1, c["ny"], c["nx"])
    f = torch.from_numpy(rng.normal(scale=0.05, size=(6,) + shape).astype(np.float32)).double().cuda()
    for q in (2, 3, 4):
        f[q, c["nz"]] = 0  # half-integer z: that plane is unused
    gam = c["gamma"]
    beta = math.sqrt(1 - 1 / gam ** 2)
    h = (1.0, 1.0, gam * (1 + beta) / 2)
    parts = []
    for sp, n in ((0, c["n"]), (1, c["ions"])):
        cells = (c["nx"], c["ny"], c["nz"] - 16)  # away from the absorbing ends
        pos = [rng.integers(0, m, n) + rng.integers(0, 1 << 20, n) / float(1 << 20) for m in cells]
        pos[2] += 8
        if c["dim"] == 2:
            pos[1] = np.zeros(n)
        u = rng.normal(scale=0.5, size=(3, n)).astype(np.float32).astype(np.float64)
        if sp == 1:
            u[:] = 0
        u[2] -= gam * beta
        w = (0.01 * c["nx"] * c["ny"] * c["nz"] / c["n"] * rng.uniform(0.5, 1.5, n)).astype(np.float32)
        parts.append((np.stack(pos), u, w.astype(np.float64)))
    return f, h, beta, parts


def _prepare_loaded(c, seed):
    f, h, beta, parts = _bring(c, seed)
    cells = c["nx"] * c["ny"] * c["nz"]
    sim = _sim(dict(c, dz=0.5), seed, slots=max(16.0, math.ceil(6.0 * max(c["n"], c["ions"]) / cells)))
    sim.set_fields({k: f[q] for q, k in enumerate(("Ex", "Ey", "Ez", "Bx", "By", "Bz"))})
    for sp, (pos, u, w) in enumerate(parts):
        if len(w):
            x = pos * np.array([[h[0]], [h[1]], [sim.sizes.hz]])
            sim.load_particles(sp, np.concatenate([x, u, w[None]]))
    s = {"case": c, "sim": sim, "eb": _fields_out(sim, 6), "cur": _fields_out(sim, 3)}
    if c["kind"] == "loaded":
        s["state"] = _checkpoint(sim)
    return s


def _prepare_batch(c, seed):
    rng = np.random.default_rng(seed)
    sims, keep, outs = [], [], []
    for r in range(c["runs"]):
        st = W.c4_run(r, (c["nz_lo"], c["nz_hi"]), c["nx"])  # the runs' boosts and lengths
        g, p, l = st.grid, st.plasma, st.laser
        sim = P.Simulation(dim=2, nx=g["nx"], nz=g["nz"], dx=g["dx"], dz=g["dz"], gamma_boost=g["gamma_boost"],
                           filter_passes=g["filter_passes"], seed=g["seed"] + 7919 * seed, slots_per_cell=8.0,
                           stream=torch.cuda.Stream())
        sim.load_plasma(p["ne"], p["z_start"], p["z_end"], p["ramp"], p["ppc"], p["jitter"],
                        [float(v) for v in rng.uniform(-0.025, 0.025, 8)], p["ions"])
        sim.launch_laser(float(rng.uniform(0.5, 2.0)), l["waist"], l["fwhm"], t_peak=0.5)
        sims.append(sim)
    batch = P.Batch(sims)
    batch.step(c["advance"])
    for sim in sims:
        keep.append(_checkpoint(sim))
        outs.append(_fields_out(sim, 6))
    return {"case": c, "batch": batch, "sims": sims, "state": keep, "eb": outs}


def _prepare_adjoint(c, seed):
    rng = np.random.default_rng(seed)
    sim = _sim(c, seed, stream=torch.cuda.Stream(), slots=8.0 if c["dim"] == 2 else 10.0)
    hz = sim.sizes.hz
    z0 = c["gamma"] * 6 * hz
    sim.load_plasma(0.001, z0, z0 + 20000.0, 2.0, _ppc(c), 0.1, [float(v) for v in rng.uniform(-0.02, 0.02, c["profile"])])
    sim.launch_laser(float(rng.uniform(0.8, 1.2)), 12.0, 8.0, t_peak=0.5)
    buffers = sim.adjoint_buffers(c["steps"], c["every"])
    cot = torch.zeros_like(buffers[1])
    k = torch.arange(c["nz"] + 1, device="cuda", dtype=torch.float32)
    mid, wid = c["steps"] * float(rng.uniform(0.25, 0.35)), 0.15 * c["steps"]  # where the light and the plasma meet
    bell = torch.exp(-((k - mid) / wid) ** 2).to(cot.dtype)
    cot[2, :, ..., c["nx"] // 2] = bell if c["dim"] == 2 else bell[:, None]  # a wake amplitude on axis
    cot[1] += 0.1 * bell.reshape((-1,) + (1,) * (c["dim"] - 1))                 # and the transmitted light
    torch.cuda.synchronize()
    return {"case": c, "sim": sim, "buffers": buffers, "cot": cot}


# -------------------------------------------------------------------- one pass


def run(s):
    c = s["case"]
    if c["kind"] == "batch":
        for sim, buf in zip(s["sims"], s["state"]):
            _restore(sim, buf)
        s["batch"].step(c["steps"])
        return [_read(sim, EB, o) for sim, o in zip(s["sims"], s["eb"])]
    sim = s["sim"]
    if c["kind"] == "adjoint":
        with torch.cuda.stream(sim.stream):
            out = sim.adjoint_forward(c["steps"], c["every"], buffers=s["buffers"])
            grad = sim.adjoint_backward(s["cot"])
        return {"fields": out, "grad": np.asarray(grad, dtype=np.float32)}
    if c["kind"] == "view":
        d = sim.diagnostics()
        return {"lab": _read(sim, EB, s["eb"], P.PIC_FRAME_LAB), "rho": sim.rho(),
                "energy": [d.field_energy, d.kinetic_energy], "count": [d.n_particles[0], d.n_particles[1]]}
    _restore(sim, s["state"])
    sim.step(c["steps"])
    out = {"eb": _read(sim, EB, s["eb"]), "j": _read(sim, CUR, s["cur"])}
    if c["gamma"] == 1.0:  # (of a neutral boosted plasma only rounding is left)
        out["rho"] = sim.rho()
    if c["dim"] == 2 or c["kind"] == "loaded":
        out["kinetic"] = sim.diagnostics().kinetic_energy
    for j, b in enumerate(s.get("snap", ())):
        P.pic_btd_get(sim.ctx, j, b.data_ptr(), b.numel() * 4, True)
    if "snap" in s:
        n = 6 * 2000 * c["nx"]
        out["lab"] = [b[:n] for b in s["snap"]]
        out["filled"] = [b[n:].view(torch.int32) for b in s["snap"]]
    return out


# ----------------------------------------------------------- the work of a pass


def work(case):
    c = case
    if c["kind"] == "batch":
        cells = c["runs"] * c["nx"] * (c["nz_lo"] + c["nz_hi"]) / 2
        c = dict(dim=2, fp64=False, kind="stage", order=1, passes=2, steps=c["steps"], gamma=13.0)
        parts = 4 * cells
    else:
        cells = c["nx"] * c["ny"] * c["nz"]
        parts = c["n"] + c["ions"] if "n" in c else cells * np.prod(_ppc(c))
        if c["kind"] == "stage" and c["gamma"] == 1.0:
            parts *= 0.8
    e = 8 if c.get("fp64") else 4
    rec = (c["dim"] + 4) * e + 4                          # offsets, weight, momentum, cell
    support = (c["order"] + 1) ** c["dim"]
    gather, push, deposit = 2 * 6 * support, 90, 3 * 4 * (c["order"] + 2) ** c["dim"]
    if c["kind"] == "view":  # fields read and written, every record read, the density written
        return {"bytes": float((6 + 6 + 1) * cells * e + parts * rec), "flops": float(parts * (support * 4 + 20))}
    # a step reads and writes every record and the fields, and writes and reads J
    bytes_ = 2 * rec * parts + (6 + 6 + 3 + 3) * e * cells
    flops = parts * (gather + push + deposit) + cells * (36 + 3 * c["dim"] * 3 * c["passes"])
    n = c["steps"]
    if c["kind"] == "adjoint":  # the forward run, and the reverse of every step (twice its operations)
        return {"bytes": float(2 * n * bytes_), "flops": float(3 * n * flops)}
    return {"bytes": float(n * bytes_), "flops": float(n * flops)}


# ------------------------------------------------------- the results in 64 bits


def exact(case, seed):
    if case["kind"] == "view":
        return _exact_view(case, seed)
    if case["kind"] == "loaded":
        return _exact_loaded(case, seed)
    return None


def _spline(p, order):
    """First node and weights (n, order + 1) of the B-spline of a position in cells."""
    if order == 1:
        b = torch.floor(p)
        d = p - b
        return b.long(), torch.stack([1 - d, d], 1)
    b = torch.floor(p + 0.5)
    d = p - b
    return b.long() - 1, torch.stack([0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2], 1)


# half-cell staggering (x, y, z) of Ex Ey Ez Bx By Bz
STAG = ((1, 0, 0), (0, 1, 0), (0, 0, 1), (0, 1, 1), (1, 0, 1), (1, 1, 0))


def _nodes(c, i, j, k):
    """Flat node index, periodic in x and y; nodes outside [0, nz] are masked."""
    ok = (k >= 0) & (k <= c["nz"])
    return (k.clamp(0, c["nz"]) * c["ny"] + j % c["ny"]) * c["nx"] + i % c["nx"], ok


def _axes(c):
    return (0, 1, 2) if c["dim"] == 3 else (0, 2)


def _support(c, pos, stag):
    """Per axis, first node and weights of a component's support (a single node along an ignorable y)."""
    out = []
    for a in range(3):
        if a in _axes(c):
            out.append(_spline(pos[a] - 0.5 * stag[a], c["order"]))
        else:
            out.append((torch.zeros_like(pos[a]).long(), torch.ones_like(pos[a])[:, None]))
    return out


def _each(sup):
    for q in range(sup[0][1].shape[1]):
        for r in range(sup[1][1].shape[1]):
            for t in range(sup[2][1].shape[1]):
                yield q, r, t


def _density(c, pos, w):
    rho = torch.zeros((c["nz"] + 1) * c["ny"] * c["nx"], dtype=torch.float64, device="cuda")
    sup = _support(c, pos, (0, 0, 0))
    for q, r, t in _each(sup):
        o, ok = _nodes(c, sup[0][0] + q, sup[1][0] + r, sup[2][0] + t)
        rho.index_add_(0, o, w * sup[0][1][:, q] * sup[1][1][:, r] * sup[2][1][:, t] * ok)
    return rho.reshape(c["nz"] + 1, c["ny"], c["nx"])


def _kinetic(u, w):
    u2 = (u * u).sum(0)
    return float((w * (u2 / (torch.sqrt(1 + u2) + 1))).sum())


def _cuda(parts):
    return [tuple(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in p) for p in parts]


def _exact_view(c, seed):
    f, h, beta, parts = _bring(c, seed)
    gam, nz = c["gamma"], c["nz"]
    vol = h[0] * h[2] * (h[1] if c["dim"] == 3 else 1.0)
    Ex, Ey, Ez, Bx, By, Bz = f

    def at_nodes(v):  # half-integer planes 0..nz-1 -> integer planes, the nearer one at the ends
        m = torch.empty_like(v)
        m[1:nz] = 0.5 * (v[:nz - 1] + v[1:nz])
        m[0], m[nz] = v[0], v[nz - 1]
        return m

    def at_halves(v):  # integer planes 0..nz -> half-integer planes
        m = torch.zeros_like(v)
        m[:nz] = 0.5 * (v[:nz] + v[1:])
        return m

    lab = torch.stack([gam * (Ex + beta * at_nodes(By)), gam * (Ey - beta * at_nodes(Bx)), Ez,
                       gam * (Bx - beta * at_halves(Ey)), gam * (By + beta * at_halves(Ex)), Bz])
    lab[2:5, nz] = 0
    (pe, ue, we), (pi, _, wi) = _cuda(parts)
    rho = (_density(c, pi, wi) - _density(c, pe, we)) / vol
    return {"lab": lab, "rho": rho, "energy": [0.5 * vol * float((f * f).sum()), _kinetic(ue, we)], "count": None}


def _exact_loaded(c, seed):
    """Explicit steps of the method: gather, Boris, Esirkepov, filter, Yee with Mur's condition."""
    f, h, _, parts = _bring(c, seed)
    f = [v.clone() for v in f]
    pos, u, w = _cuda(parts[:1])[0]
    nx, ny, nz, S = c["nx"], c["ny"], c["nz"], c["order"]
    ax3 = c["dim"] == 3
    dt = 0.99 / math.sqrt(sum(1 / h[a] ** 2 for a in _axes(c)))
    vol = h[0] * h[2] * (h[1] if ax3 else 1.0)
    eps = -math.pi * dt
    rot = {0: 2, 1: 1, 2: 0}  # axis -> tensor dimension
    for _ in range(c["steps"]):
        eb = []
        for q in range(6):
            sup = _support(c, pos, STAG[q])
            v = torch.zeros_like(w)
            flat = f[q].reshape(-1)
            for a, b, t in _each(sup):
                o, ok = _nodes(c, sup[0][0] + a, sup[1][0] + b, sup[2][0] + t)
                v += flat[o] * ok * sup[0][1][:, a] * sup[1][1][:, b] * sup[2][1][:, t]
            eb.append(v)
        e, b = torch.stack(eb[:3]), torch.stack(eb[3:])
        um = u + eps * e
        t = eps * b / torch.sqrt(1 + (um * um).sum(0))
        s = 2 * t / (1 + (t * t).sum(0))
        up = um + torch.linalg.cross(um, t, dim=0)
        u = um + torch.linalg.cross(up, s, dim=0) + eps * e
        v = u / torch.sqrt(1 + (u * u).sum(0))
        new = pos.clone()
        for a in _axes(c):
            new[a] = pos[a] + dt * v[a] / h[a]
        cur = _esirkepov(c, pos, new, w, v[1], dt, h, vol)
        pos = new
        for _p in range(c["passes"]):
            for a in _axes(c):
                d = rot[a]
                for q in range(3):
                    if a == 2:
                        z = torch.zeros_like(cur[q][:1])
                        top = nz if q == 2 else nz + 1
                        x = cur[q][:top]
                        x = 0.5 * x + 0.25 * (torch.cat([z, x[:-1]]) + torch.cat([x[1:], z]))
                        cur[q] = torch.cat([x, cur[q][top:]])
                    else:
                        cur[q] = 0.5 * cur[q] + 0.25 * (cur[q].roll(1, d) + cur[q].roll(-1, d))
        _yee(c, f, cur, dt, h, ax3)
        pos[0] %= nx
        if ax3:
            pos[1] %= ny
    return {"eb": torch.stack(f), "j": torch.stack(cur), "rho": -_density(c, pos, w) / vol, "kinetic": _kinetic(u, w)}


def _esirkepov(c, p0, p1, w, vy, dt, h, vol):
    """Charge-conserving current of the moves p0 -> p1 (electrons)."""
    S = c["order"]
    n = p0.shape[1]
    first, s0, ds = [], [], []
    for a in range(3):
        if a not in _axes(c):
            first.append(torch.zeros(n, dtype=torch.long, device="cuda"))
            s0.append(torch.ones(n, 1, dtype=torch.float64, device="cuda"))
            ds.append(torch.zeros(n, 1, dtype=torch.float64, device="cuda"))
            continue
        (b0, w0), (b1, w1) = _spline(p0[a], S), _spline(p1[a], S)
        b = torch.minimum(b0, b1)
        g0, g1 = (torch.zeros(n, S + 2, dtype=torch.float64, device="cuda") for _ in range(2))
        for q in range(S + 1):
            g0.scatter_(1, (b0 - b + q)[:, None], w0[:, q:q + 1])
            g1.scatter_(1, (b1 - b + q)[:, None], w1[:, q:q + 1])
        first.append(b)
        s0.append(g0)
        ds.append(g1 - g0)
    cur = [torch.zeros((c["nz"] + 1) * c["ny"] * c["nx"], dtype=torch.float64, device="cuda") for _ in range(3)]
    m = [s.shape[1] for s in s0]
    run_ = [torch.cumsum(d, 1) for d in ds]

    def cross(a, b, i, j):  # the mean over the path of the product of two shapes
        return (s0[a][:, i] * s0[b][:, j] + 0.5 * (ds[a][:, i] * s0[b][:, j] + s0[a][:, i] * ds[b][:, j])
                + ds[a][:, i] * ds[b][:, j] / 3)

    for i in range(m[0]):
        for j in range(m[1]):
            for k in range(m[2]):
                o, ok = _nodes(c, first[0] + i, first[1] + j, first[2] + k)
                ww = w * ok
                cur[0].index_add_(0, o, h[0] / (dt * vol) * ww * run_[0][:, i] * cross(1, 2, j, k))
                if c["dim"] == 3:
                    cur[1].index_add_(0, o, h[1] / (dt * vol) * ww * run_[1][:, j] * cross(2, 0, k, i))
                else:
                    cur[1].index_add_(0, o, -ww * vy / vol * cross(0, 2, i, k))
                cur[2].index_add_(0, o, h[2] / (dt * vol) * ww * run_[2][:, k] * cross(0, 1, i, j))
    return [v.reshape(c["nz"] + 1, c["ny"], c["nx"]) for v in cur]


def _yee(c, f, cur, dt, h, ax3):
    nz = c["nz"]

    def dp(v, a):  # forward difference along x or y
        return (v.roll(-1, 2 - a) - v) / h[a] if a != 1 or ax3 else torch.zeros_like(v)

    def dm(v, a):  # backward difference
        return (v - v.roll(1, 2 - a)) / h[a] if a != 1 or ax3 else torch.zeros_like(v)

    def half_b():
        Ex, Ey, Ez, Bx, By, Bz = f
        Bx[:nz] -= 0.5 * dt * (dp(Ez, 1)[:nz] - (Ey[1:] - Ey[:nz]) / h[2])
        By[:nz] -= 0.5 * dt * ((Ex[1:] - Ex[:nz]) / h[2] - dp(Ez, 0)[:nz])
        Bz -= 0.5 * dt * (dp(Ey, 0) - dp(Ex, 1))

    half_b()
    Ex, Ey, Ez, Bx, By, Bz = f
    old = [v[[0, 1, nz - 1, nz]].clone() for v in (Ex, Ey)]
    tp = 2 * math.pi
    i = slice(1, nz)
    Ex[i] += dt * (dm(Bz, 1)[i] - (By[1:nz] - By[:nz - 1]) / h[2] - tp * cur[0][i])
    Ey[i] += dt * ((Bx[1:nz] - Bx[:nz - 1]) / h[2] - dm(Bz, 0)[i] - tp * cur[1][i])
    Ez[:nz] += dt * (dm(By, 0) - dm(Bx, 1) - tp * cur[2])[:nz]
    cm = (dt - h[2]) / (dt + h[2])
    for v, o in zip((Ex, Ey), old):
        v[0] = o[1] + cm * (v[1] - o[0])
        v[nz] = o[2] + cm * (v[nz - 1] - o[3])
    half_b()
