"""Kernels at the sizes where their splits end: the field marches (strips of 28
to 31 columns, chunks of a few planes, rows of a CTA), the restore (runs of 128
records, snapshots the device can and cannot read in place), the diagnostic
sums and the injection's quotients.  Field kernels against the FP64 oracle with
the single-phase tolerances; sums and positions against exact arithmetic."""
import math

import numpy as np
import pytest

from pairs import field_maxrel, make_pair, set_fields_both
from paper_1011_0917_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FP32, FP64 = 0, 1
# one phase on random inputs: a node is a sum of some tens of terms, each
# rounded once (the bound of the single-phase parity tests)
TOL = {FP32: 2e-6, FP64: 1e-12}


@pytest.fixture(scope="module")
def O():
    import oracle.oracle as O
    O.build_oracle()
    return O


SIZES_2D = [(1, 4), (3, 9), (28, 21), (29, 40), (31, 67), (64, 133)]
SIZES_3D = [(1, 1, 5), (5, 3, 9), (28, 29, 14), (30, 13, 40), (61, 14, 21)]


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("size", SIZES_2D + SIZES_3D)
def test_field_marches(O, size, bc, prec):
    dim = 2 if len(size) == 2 else 3
    for npass in (1, 2, 3, 4):
        g = dict(dim=dim, nx=size[0], nz=size[-1], dx=0.7, dz=0.9, filter_passes=npass, bc_z=bc, seed=1)
        if dim == 3:
            g.update(ny=size[1], dy=0.8)
        sim, o = make_pair(O, g, prec)
        shape = (size[-1] + 1, size[1] if dim == 3 else 1, size[0])
        f = {c: v for c, v in W.random_fields(shape, seed=7 + npass).items() if npass == 1 or c[0] == "J"}
        set_fields_both(sim, o, f, bc)
        sim.step_phases(16)
        o.step_phases(O.PH_FILTER)
        err = field_maxrel(sim, o, ("Jx", "Jy", "Jz"), bc)
        assert max(err.values()) < TOL[prec], (npass, err)
        if npass == 1:
            for _ in range(2):
                sim.step_phases(32)
                o.step_phases(O.PH_YEE)
            err = field_maxrel(sim, o, ("Ex", "Ey", "Ez", "Bx", "By", "Bz"), bc)
            assert max(err.values()) < TOL[prec], err
        sim.close()


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("ids", [False, True])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 5000])
def test_restore_in_place_and_staged(n, ids, prec):
    import torch

    import paper_1011_0917_gb300 as P
    kw = dict(dim=2, nx=40, nz=50, dx=1.0, dz=0.5, gamma_boost=5.0, precision=prec, track_ids=ids, slots_per_cell=16.0)
    sim = P.Simulation(**kw)
    st = W.random_particles(n, (40.0, 1.0, 49.0 * sim.sizes.hz), seed=n, u_scale=0.3)
    st[5] -= 5.0 * sim.sizes.beta
    sim.load_particles(0, st, np.arange(n) * 3)
    sim.load_particles(1, st[:, : max(1, n // 2)], np.arange(max(1, n // 2)) * 3)
    nb = P.pic_state_bytes(sim.ctx)
    # at byte offsets 0 and 4 of device memory (the second misaligns FP64
    # columns), and in host memory
    dev = torch.zeros(nb + 4, dtype=torch.uint8, device="cuda")
    want = []
    for sp in (0, 1):
        a, i = sim.particles(sp, with_ids=ids)
        want.append(a[:, np.lexsort(a)])
    for off in (0, 4, None):
        other = P.Simulation(**kw)
        if off is None:
            host = np.zeros(nb, dtype=np.uint8)
            P.pic_get_state(sim.ctx, host.ctypes.data, nb, False)
            P.pic_set_state(other.ctx, host.ctypes.data, nb, False)
        else:
            P.pic_get_state(sim.ctx, dev.data_ptr() + off, nb, True)
            P.pic_set_state(other.ctx, dev.data_ptr() + off, nb, True)
        for sp in (0, 1):
            a, i = other.particles(sp, with_ids=ids)
            assert np.array_equal(a[:, np.lexsort(a)], want[sp]), (off, sp)
            if ids:
                b, j = sim.particles(sp, with_ids=True)
                assert np.array_equal(np.sort(i), np.sort(j))
        other.close()


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("nx,nz,n", [(3, 5, 2), (40, 90, 33), (200, 300, 60000)])
def test_sums_are_exact(nx, nz, n, prec):
    """Energies and charge of resting and moving records and random fields
    (tiny, huge and zero values among them) against exact sums: FP64's last
    bits, a few of them for the final products."""
    import torch

    import paper_1011_0917_gb300 as P
    sim = P.Simulation(dim=2, nx=nx, nz=nz, dx=1.0, dz=1 / 32, gamma_boost=13.0, precision=prec, slots_per_cell=64.0)
    rng = np.random.default_rng(nx)
    real = np.float32 if prec == FP32 else np.float64
    f = {}
    for c in ("Ex", "Ey", "Ez", "Bx", "By", "Bz"):
        v = rng.normal(scale=0.05, size=(nz + 1, 1, nx)).astype(real)
        v.ravel()[::7] = 0
        v.ravel()[::11] *= real(1e-20)
        if c in ("Ez", "Bx", "By"):
            v[nz] = 0
        f[c] = v
    if n == 2:
        f["Ex"].ravel()[1] = real(3e15)
    sim.set_fields({c: torch.from_numpy(v) for c, v in f.items()})
    U = float(real(-13.0 * sim.sizes.beta))
    st = np.zeros((7, n))
    st[0] = rng.uniform(0, nx, n)
    st[2] = rng.uniform(0, 0.99 * nz * sim.sizes.hz, n)
    du = rng.normal(scale=0.3, size=(3, n)).astype(np.float32).astype(np.float64)
    du[:, ::2] = 0
    st[3:6] = du
    st[5] += U
    st[6] = rng.uniform(0.5, 1.5, n).astype(np.float32)
    sim.load_particles(0, st)
    sim.load_particles(1, st[:, : n // 2 + 1])
    d = sim.diagnostics()
    want = 0.5 * sim.sizes.hz * math.fsum(float(x) ** 2 for v in f.values() for x in v.ravel())
    assert abs(d.field_energy / want - 1) < 1e-15
    L = np.longdouble
    dz = (st[5] - U).astype(real).astype(np.float64)  # as stored
    u2 = L(du[0]) ** 2 + L(du[1]) ** 2 + (L(dz) + L(U)) ** 2
    want = float(np.sum(L(st[6]) * (u2 / (np.sqrt(1 + u2) + 1))))
    assert abs(d.kinetic_energy / want - 1) < 1e-15
    want = math.fsum(st[6][: n // 2 + 1]) - math.fsum(st[6])
    assert abs(d.charge - want) < 1e-15 * math.fsum(st[6])
    assert (d.n_particles[0], d.n_particles[1], d.n_paired) == (n, n // 2 + 1, 0)


@pytest.mark.parametrize("dim,h,ppc,gamma", [(2, 0.7, (3, 1, 2), 1.0), (2, 1 / 3, (2, 1, 5), 13.0), (3, 0.9, (2, 3, 2), 5.0)])
def test_lattice_positions_bit_for_bit(dim, h, ppc, gamma):
    """Loaded electrons at x = cell h + offset h of the lattice formula in IEEE
    doubles (quotients correctly rounded): the FP64 positions bit for bit."""
    import paper_1011_0917_gb300 as P
    seed, jit = 77, 0.17
    nx, ny, nz = 11, (7 if dim == 3 else 1), 23
    sim = P.Simulation(dim=dim, nx=nx, ny=ny, nz=nz, dx=h, dy=1.1 * h, dz=0.13, gamma_boost=gamma, precision=FP64, seed=seed,
                       slots_per_cell=80.0, track_ids=True)
    s = sim.sizes
    z0 = 0.31
    sim.load_plasma(0.01, z0, z0 + 40.0, 0.0, ppc, jit)
    got, ids = sim.particles(0, with_ids=True)
    M = (1 << 64) - 1

    def uniform(counter):
        z = (seed + (counter + 1) * 0x9E3779B97F4A7C15) & M
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M
        return float((z ^ (z >> 31)) >> 11) * (1.0 / 9007199254740992.0)

    def place(x, hh, n):
        xi = x / hh
        c = math.floor(xi)
        return (float(c % n) + (xi - float(c))) * hh

    gam, hz = gamma, s.hz
    NX, NY = nx * ppc[0], (ny * ppc[1] if dim == 3 else 1)
    hzl = gam * hz
    dzl = hzl / float(ppc[2])
    assert len(ids) > 0
    for q in range(0, len(ids), 7):
        i = int(ids[q])
        ix, iy, m = i % NX, (i // NX) % NY, i // (NX * NY)
        x = (float(ix) + 0.5) * (s.hx / float(ppc[0])) + (jit * s.hx) * (2.0 * uniform(3 * i) - 1.0)
        x = x + nx * s.hx if x < 0 else x
        x = x - nx * s.hx if x >= nx * s.hx else x
        assert got[0, q] == place(x, s.hx, nx)
        if dim == 3:
            y = (float(iy) + 0.5) * (s.hy / float(ppc[1])) + (jit * s.hy) * (2.0 * uniform(3 * i + 1) - 1.0)
            y = y + ny * s.hy if y < 0 else y
            y = y - ny * s.hy if y >= ny * s.hy else y
            assert got[1, q] == place(y, s.hy, ny)
        z = z0 + (float(m) + 0.5) * dzl + (jit * hzl) * (2.0 * uniform(3 * i + 2) - 1.0)
        assert got[2, q] == place(z / gam, hz, nz)  # (at t = 0, no window)
