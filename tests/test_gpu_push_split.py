"""The push with several CTAs per tile (grids of few tiles) and with one: grids
on both sides of the line, a tile whose records leave on all sides, against the
FP64 oracle with the tolerances of the other push tests; and plasma that drifts
with its ions, whose currents cancel whichever CTA deposits a record."""
import numpy as np
import pytest

from pairs import gpu_fields, make_pair
from test_gpu_push_blocks import FP32, FP64, O, test_leavers_of_one_tile as leavers  # noqa: F401

pytestmark = pytest.mark.gpu

# tiles: 2D 16 x 16 cells, 3D 8 x 8 x 8: 56 and 289, 36, 144 and 180 (152 SMs:
# the line is at 228 tiles in 2D FP32 and at 152 otherwise)
GRIDS = [dict(dim=2, nx=112, nz=128, dx=1.0, dz=1.0, filter_passes=1, seed=3),
         dict(dim=2, nx=272, nz=272, dx=1.0, dz=1.0, filter_passes=1, seed=3),
         dict(dim=3, nx=24, ny=24, nz=32, dx=1.0, dy=1.0, dz=1.0, filter_passes=1, seed=4),
         dict(dim=3, nx=48, ny=48, nz=32, dx=1.0, dy=1.0, dz=1.0, filter_passes=1, seed=4),
         dict(dim=3, nx=48, ny=48, nz=40, dx=1.0, dy=1.0, dz=1.0, filter_passes=1, seed=4)]


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("g", GRIDS)
@pytest.mark.parametrize("shape,rel", [(1, 2), (2, 1)])
@pytest.mark.parametrize("n", [129, 1100])
def test_leavers(O, g, shape, rel, n, prec):  # noqa: F811
    leavers(O, g, shape, 0, rel, n, prec)


@pytest.mark.parametrize("g", GRIDS)
@pytest.mark.parametrize("shape,rel", [(1, 2), (2, 2), (1, 1)])
def test_electrons_and_ions_cancel(O, g, shape, rel):  # noqa: F811
    # an electron on each ion, both drifting: 700 pairs in one tile, so that a
    # pair's two records are deposited by different CTAs.  A record's deposit
    # takes at most 8 roundings of 2^-24 of it (5e-7) and the deposits on a
    # node have one sign: what is left of both is below 1e-6 of the ions'
    # current; twice that is allowed.
    g = dict(g, shape_order=shape, bc_z=0, gamma_boost=5.0, dx=1.0, dz=0.1)
    rng = np.random.default_rng(9)
    st = np.zeros((7, 700))
    st[0] = rng.uniform(16.0, 24.0, 700)
    if g["dim"] == 3:
        st[1] = rng.uniform(8.0, 16.0, 700)
    st[2] = rng.uniform(1.6, 2.4, 700)
    st[5] = -np.sqrt(5.0 ** 2 - 1.0)
    st[6] = 1.0
    both, _ = make_pair(O, g, FP32, explicit_ions=True, z_relative=rel)
    ions, _ = make_pair(O, g, FP32, explicit_ions=True, z_relative=rel)
    both.load_particles(0, st)
    for sim in (both, ions):
        sim.load_particles(1, st[:, ::-1].copy())
    for _ in range(3):
        for sim in (both, ions):
            sim.step_phases(1 | 2 | 4)
        Jb, Ji = gpu_fields(both), gpu_fields(ions)
        top = np.abs(Ji["Jz"]).max()
        assert top > 0
        for c in ("Jx", "Jy", "Jz"):
            assert np.abs(Jb[c]).max() <= 2e-6 * top, c
