"""The push with one CTA per tile, as grids of many tiles run it: whole steps
with the laser in the plasma, paired, released and explicit ions, both shapes,
both precisions and records in relative form, against the FP64 oracle.  And,
with one and with several CTAs per tile, what the current tile owes to exact
sums: an electron on its ion leaves no current, and of two that part the small
difference keeps its digits."""
import math

import numpy as np
import pytest

from pairs import field_errors, gpu_fields, make_pair, vector_errors

pytestmark = pytest.mark.gpu

FP32, FP64 = 0, 1
TOL = {FP32: 1e-4, FP64: 1e-10}  # 50 steps or fewer, as in the other full-step windows
GAM = 13.0
HZ = (1 / 32) * GAM * (1 + math.sqrt(1 - 1 / GAM ** 2))
# 288 tiles of 8 x 8 x 8, 256 of 16 x 16
BOOST3 = dict(dim=3, nx=48, ny=48, nz=64, dx=1.0, dy=1.0, dz=1 / 32, gamma_boost=GAM, filter_passes=2, seed=19)
BOOST2 = dict(dim=2, nx=128, nz=512, dx=1.0, dz=1 / 32, gamma_boost=GAM, filter_passes=2, seed=17)
RUNS = {2: (25, dict(ne=0.004, z_start=GAM * 10 * HZ, z_end=GAM * 900 * HZ, ramp=2.0, ppc=(1, 1, 2), jitter=0.1, ions=1),
            dict(a0=4.0, waist=24.0, fwhm=2.0, t_peak=0.5)),
        3: (10, dict(ne=0.004, z_start=GAM * 6 * HZ, z_end=GAM * 200 * HZ, ramp=2.0, ppc=(1, 1, 2), jitter=0.1, ions=1),
            dict(a0=4.0, waist=12.0, fwhm=2.0, t_peak=0.5))}
ORACLES = {}


@pytest.fixture(scope="module")
def O():
    import oracle.oracle as O
    O.build_oracle()
    yield O
    ORACLES.clear()


def whole_tiles(sim):
    """no tile of this grid is shared by CTAs, whatever the card's SM count"""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return sim.sizes.ntiles >= sms and 4 * sim.sizes.ntiles > 6 * sms


@pytest.mark.parametrize("prec", [FP64, FP32])
@pytest.mark.parametrize("explicit,rel", [(False, 2), (True, 2), (False, 1), (True, 1)])
@pytest.mark.parametrize("dim,shape", [(2, 1), (2, 2), (3, 1), (3, 2)])
def test_boosted_steps(O, dim, shape, explicit, rel, prec):
    g = dict(BOOST2 if dim == 2 else BOOST3, shape_order=shape)
    steps, p, laser = RUNS[dim]
    sim, o = make_pair(O, g, prec, track_ids=False, explicit_ions=explicit, z_relative=rel, slots_per_cell=8.0)
    assert whole_tiles(sim)
    if (dim, shape) not in ORACLES:
        o.load_plasma(O.PlasmaParams(**p))
        o.set_laser(O.LaserParams(pol=1, **laser))
        o.step(steps)
        ORACLES[dim, shape] = o
    o = ORACLES[dim, shape]
    sim.load_plasma(p["ne"], p["z_start"], p["z_end"], p["ramp"], p["ppc"], p["jitter"], (), p["ions"])
    sim.launch_laser(laser["a0"], laser["waist"], laser["fwhm"], 0.0, laser["t_peak"], 1)
    sim.step(steps)
    err = vector_errors(sim, o)
    assert max(err.values()) < TOL[prec], err
    # the plasma's own Ez, far below the laser's Ey, by itself
    assert np.abs(o.field("Ez")).max() > 1e-6 * np.abs(o.field("Ey")).max()
    assert field_errors(sim, o, ("Ez",))["Ez"] < TOL[prec]
    d = sim.diagnostics()
    assert d.n_particles[0] == o.num(0) and d.n_particles[1] == o.num(1)
    assert d.n_paired == 0 if explicit else 0 < d.n_paired < d.n_particles[0]
    sim.close()


GRIDS = [dict(dim=2, nx=48, nz=64), dict(dim=2, nx=272, nz=272), dict(dim=3, nx=24, ny=24, nz=24),
         dict(dim=3, nx=48, ny=48, nz=64)]


@pytest.mark.parametrize("g", GRIDS)
@pytest.mark.parametrize("shape,rel,explicit", [(1, 2, False), (2, 2, False), (1, 1, False), (1, 1, True), (2, 1, True)])
def test_an_electron_on_its_ion_leaves_no_current(O, g, shape, rel, explicit):
    # 700 pairs in one tile, an electron's record and its ion's at different
    # places of their lists, both drifting with the FP32 drift momentum.  The
    # ions are in the electrons' kernel here (records in relative form, or not
    # explicit ions), so both deposits are sums of the same integers.
    g = dict(g, dx=1.0, dy=1.0, dz=0.1, shape_order=shape, bc_z=0, gamma_boost=5.0, filter_passes=1, seed=4)
    rng = np.random.default_rng(9)
    both, _ = make_pair(O, g, FP32, explicit_ions=explicit, z_relative=rel)
    ions, _ = make_pair(O, g, FP32, explicit_ions=explicit, z_relative=rel)
    st = np.zeros((7, 700))
    st[0] = rng.uniform(16.0, 24.0, 700)
    if g["dim"] == 3:
        st[1] = rng.uniform(8.0, 16.0, 700)
    st[2] = rng.uniform(1.6, 2.4, 700)
    st[5] = float(np.float32(-5.0 * both.sizes.beta))
    st[6] = rng.uniform(0.5, 1.5, 700)
    both.load_particles(0, st)
    for sim in (both, ions):
        sim.load_particles(1, st[:, ::-1].copy())
    for _ in range(4):
        for sim in (both, ions):
            sim.step_phases(1 | 2 | 4)
        Jb, Ji = gpu_fields(both), gpu_fields(ions)
        assert np.abs(Ji["Jz"]).max() > 0
        for c in ("Jx", "Jy", "Jz"):
            assert not Jb[c].any(), (c, np.abs(Jb[c]).max() / np.abs(Ji["Jz"]).max())


@pytest.mark.parametrize("g", GRIDS)
@pytest.mark.parametrize("shape", [1, 2])
def test_current_of_parting_pairs(O, g, shape):
    # gamma = 130, electrons pushed off their ions by du ~ 0.3: the current
    # along z is the difference of two that are some 1000 times larger.
    # An electron's departure takes at most 6 roundings of 2^-24, its node's
    # sum 3 more on the way to J: below 1e-6 of the current in all.  The words
    # of the current tile add 2^-39 of a largest deposit per contribution
    # (tiles of 1024 slots and their ions: scale 2^19, 19 further bits), of
    # which a node takes fewer than 200.  FP32 deposits (2^-24 of each of two
    # large currents) would be off by 50 times as much.
    g = dict(g, dx=1.0, dy=1.0, dz=0.03, shape_order=shape, bc_z=0, gamma_boost=130.0, filter_passes=1, seed=4)
    sim, o = make_pair(O, g, FP32, explicit_ions=True, z_relative=1, slots_per_cell=2.0)
    size = (g["nx"], g.get("ny", 1), g["nz"])
    rng = np.random.default_rng(5)
    n = 3000
    st = np.zeros((7, n))
    for q, h in ((0, 1.0), (1, 1.0), (2, o.hz)):
        if q != 1 or g["dim"] == 3:  # offsets that FP32 holds
            st[q] = (rng.integers(0, size[q], n) + rng.integers(0, 1 << 20, n) / 2.0 ** 20) * h
    U = float(np.float32(-130.0 * o.beta))
    du = rng.normal(scale=0.3, size=(3, n)).astype(np.float32).astype(np.float64)
    w = rng.uniform(0.5, 1.0, n).astype(np.float32).astype(np.float64)
    for sp in (0, 1):
        s = st.copy()
        if sp == 0:
            s[3:6] = du
        s[5] += U
        s[6] = w
        ids = np.arange(n, dtype=np.int64)
        sim.load_particles(sp, s, ids)
        o.add_particles(sp, s[0], s[1], s[2], s[3], s[4], s[5], s[6], ids)
    sim.step_phases(1 | 2 | 4)
    o.step_phases(O.PH_ZERO_J | O.PH_PUSH | O.PH_IONS)
    J = gpu_fields(sim)
    vol = o.hz
    for c, f in (("Jx", 1.0 / (o.dt * vol)), ("Jy", 1.0 / (o.dt * vol) if g["dim"] == 3 else 1.0 / vol),
                 ("Jz", o.hz / (o.dt * vol))):
        want = o.field(c)[:g["nz"]]
        top = np.abs(want).max()
        assert top > 0
        if c == "Jz":
            assert top < 0.02 * f
        err = np.abs(J[c][:g["nz"]] - want).max()
        assert err <= 1e-6 * top + 200 * 2.0 ** -39 * f, (c, err / top, top / f)
