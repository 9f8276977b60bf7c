"""Values at the ends of the working precision in the calls that read results:
infinities, NaN and values whose sums leave the range in the lab-frame view,
weights whose sums leave it in the diagnostics, against FP64."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FP32, FP64 = 0, 1


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("gam", [1.5, 13.0, 130.0])
@pytest.mark.parametrize("dim", [2, 3])
def test_lab_view_of_extreme_fields(dim, gam, prec):
    import torch

    import paper_1011_0917_gb300 as P
    nx, ny, nz = 8, (3 if dim == 3 else 1), 64
    sim = P.Simulation(dim=dim, nx=nx, ny=ny, nz=nz, dx=1.0, dy=1.0, dz=0.1, gamma_boost=gam, precision=prec)
    real = np.float32 if prec == FP32 else np.float64
    rng = np.random.default_rng(1)
    big = real(3e38) if prec == FP32 else real(1.5e308)
    F = {}
    for c in ("Ex", "Ey", "Ez", "Bx", "By", "Bz"):
        v = rng.normal(size=(nz + 1, ny, nx)).astype(real)
        r = v.ravel()
        r[::13], r[5::17], r[3::19] = np.inf, -np.inf, np.nan
        r[7::23], r[11::29], r[2::31] = big, -big, 0
        r[4::37] *= real(1e-30)
        if c in ("Ez", "Bx", "By"):
            v[nz] = 0
        F[c] = v
    sim.set_fields({c: torch.from_numpy(v) for c, v in F.items()})
    got = {c: t.cpu().numpy().reshape(nz + 1, ny, nx) for c, t in sim.fields(0x3F, frame=1).items()}
    b = sim.sizes.beta
    with np.errstate(all="ignore"):
        D = {c: v.astype(np.float64) for c, v in F.items()}

        def at_nodes(v):
            return np.concatenate([0.5 * (v[:1] + v[:1]), 0.5 * (v[:nz - 1] + v[1:nz]), 0.5 * (v[nz - 1:nz] + v[nz - 1:nz])])

        def at_halves(v):
            return np.concatenate([0.5 * (v[:nz] + v[1:]), np.zeros_like(v[:1])])

        for c, p, sign, mean in (("Ex", "By", 1, at_nodes), ("Ey", "Bx", -1, at_nodes), ("Bx", "Ey", -1, at_halves),
                                 ("By", "Ex", 1, at_halves)):
            m = mean(D[p])
            want = (gam * (D[c] + (sign * b) * m)).astype(real)
            if mean is at_halves:
                want[nz] = 0
            g = got[c]
            finite = np.isfinite(want)
            assert np.array_equal(np.isnan(g), np.isnan(want)), c
            assert np.array_equal(g[~finite & ~np.isnan(want)], want[~finite & ~np.isnan(want)]), c
            if prec == FP64:
                assert np.array_equal(g[finite], want[finite]), c
            else:
                # one rounding, after at most eight operations on pairs good to
                # 2^-46 of their larger operand each
                bound = np.spacing(np.abs(want)) + gam * 2.0 ** -43 * (np.abs(D[c]) + np.abs(m))
                assert (np.abs(g.astype(np.float64) - want)[finite] <= bound[finite]).all(), c
        for c in ("Ez", "Bz"):
            assert np.array_equal(got[c], F[c], equal_nan=True), c


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("w", [1e29, 3e30, 3e38])
def test_sums_of_huge_weights(w, prec):
    # 3000 records in one tile, half of them at rest relative to the drift: a
    # thread adds a dozen of them before its sum is carried over to FP64
    import paper_1011_0917_gb300 as P
    sim = P.Simulation(dim=2, nx=16, nz=16, dx=1.0, dz=0.1, gamma_boost=5.0, precision=prec, slots_per_cell=16.0)
    real = np.float32 if prec == FP32 else np.float64
    rng = np.random.default_rng(2)
    n = 3000
    U = float(real(-5.0 * sim.sizes.beta))
    st = np.zeros((7, n))
    st[0], st[2] = rng.uniform(0.0, 16.0, n), rng.uniform(0.0, 15.9, n) * sim.sizes.hz
    st[3, ::2] = rng.normal(size=n // 2).astype(np.float32)
    st[5] = U
    st[6] = (w * rng.uniform(0.5, 1.0, n)).astype(real)
    sim.load_particles(0, st)
    d = sim.diagnostics()
    want = math.fsum(st[6])
    assert abs(d.charge + want) <= 1e-15 * want
    u2 = np.longdouble(st[3]) ** 2 + np.longdouble(U) ** 2
    want = float(np.sum(np.longdouble(st[6]) * (u2 / (np.sqrt(1 + u2) + 1))))
    assert abs(d.kinetic_energy - want) <= 1e-15 * want
