"""The push where its blocks of 32 records and its queues of 32 leavers end:
particle counts around those sizes, all of them at the edges of one tile and
moving fast, so that a warp's records leave for several tiles at once (through
the periodic ends and a ragged last tile too).  Particles by id and currents
against the FP64 oracle, with the tolerances of the single-phase tests."""
import numpy as np
import pytest

from pairs import field_maxrel, gpu_particles, make_pair, oracle_particles, periodic_delta

pytestmark = pytest.mark.gpu

FP32, FP64 = 0, 1
POS = {FP32: 2e-6, FP64: 1e-12}
CUR = {FP32: 1e-5, FP64: 1e-12}
G2 = dict(dim=2, nx=24, nz=40, dx=1.0, dz=1.0, filter_passes=1, seed=3)
G3 = dict(dim=3, nx=12, ny=10, nz=20, dx=1.0, dy=1.0, dz=1.0, filter_passes=1, seed=4)


@pytest.fixture(scope="module")
def O():
    import oracle.oracle as O
    O.build_oracle()
    return O


def _same_particles(sim, o, sp, prec, bc):
    a, ia = gpu_particles(sim, sp)
    b, ib = oracle_particles(o, sp)
    assert np.array_equal(ia, ib), (sp, len(ia), len(ib))
    for q, L, h in ((0, o.Lx, o.hx), (1, o.Ly, o.hy), (2, o.Lz, o.hz)):
        d = np.abs(periodic_delta(a[q], b[q], L) if q < 2 or bc == 0 else a[q] - b[q]) / h
        assert len(d) == 0 or d.max() < POS[prec], (q, d.max())


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("g,shape,bc,rel", [(G2, 1, 1, 2), (G2, 2, 0, 2), (G2, 1, 0, 1), (G3, 1, 0, 2), (G3, 1, 1, 1),
                                            (G3, 2, 1, 2)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 257, 1300])
def test_leavers_of_one_tile(O, g, shape, bc, rel, n, prec):
    g = dict(g, shape_order=shape, bc_z=bc)
    sim, o = make_pair(O, g, prec, z_relative=rel)
    rng = np.random.default_rng(100 + n)
    edge = (16, 0, 16) if g["dim"] == 2 else (8, 8, 8)  # the ragged tile's lower corner
    size = (g["nx"], g.get("ny", 1), g["nz"])
    st = np.zeros((7, n))
    for q in range(3):
        if q == 1 and g["dim"] == 2:
            continue
        # within a quarter cell of the tile's lower face or of its upper end
        hi = min(size[q], edge[q] + (16 if g["dim"] == 2 else 8))
        low = edge[q] + rng.uniform(0.0, 0.25, n)
        st[q] = np.where(rng.random(n) < 0.5, low, hi - rng.uniform(0.01, 0.25, n))
        if bc == 1 and q == 2:
            st[q] = low  # (not out of the box)
    st[3:6] = rng.choice([-3.0, 3.0], size=(3, n))
    st[6] = rng.uniform(0.5, 1.5, n)
    ids = np.arange(n, dtype=np.int64) * 5 + 2
    sim.load_particles(0, st, ids)
    o.add_particles(0, st[0], st[1], st[2], st[3], st[4], st[5], st[6], ids)
    for _ in range(2):
        sim.step_phases(1 | 2)
        o.step_phases(O.PH_ZERO_J | O.PH_PUSH)
    _same_particles(sim, o, 0, prec, bc)
    err = field_maxrel(sim, o, ("Jx", "Jy", "Jz"), bc)
    assert max(err.values()) < CUR[prec], err


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("g,bc", [(G2, 1), (G2, 0), (G3, 1), (G3, 0)])
@pytest.mark.parametrize("n", [1, 32, 33, 900])
def test_ions_of_one_layer_leave(O, g, bc, n, prec):
    # every ion sits on the lowest cells of the bottom or the second tile
    # layer and drifts down: all of them leave their tile in one step
    g = dict(g, bc_z=bc, gamma_boost=5.0, dz=0.1)
    sim, o = make_pair(O, g, prec, explicit_ions=True)
    rng = np.random.default_rng(200 + n)
    st = np.zeros((7, n))
    st[0] = rng.uniform(0, o.Lx, n)
    if g["dim"] == 3:
        st[1] = rng.uniform(0, o.Ly, n)
    layer = 16 if g["dim"] == 2 else 8
    st[2] = (np.where(rng.random(n) < 0.5, 0, layer) + rng.uniform(0.0, 0.2, n)) * o.hz
    st[5] = -5.0 * o.beta
    st[6] = rng.uniform(0.5, 1.5, n)
    ids = np.arange(n, dtype=np.int64)
    sim.load_particles(1, st, ids)
    o.add_particles(1, st[0], st[1], st[2], st[3], st[4], st[5], st[6], ids)
    for _ in range(2):
        sim.step_phases(1 | 4)
        o.step_phases(O.PH_ZERO_J | O.PH_IONS)
    _same_particles(sim, o, 1, prec, bc)
    err = field_maxrel(sim, o, ("Jz",), bc)
    assert max(err.values()) < CUR[prec], err
