"""The kernel launches that pic_profile_read reports, where a phase's work is
done by a kernel on some grids and by a memset on others."""
import pytest

pytestmark = pytest.mark.gpu


# zeroing J: a kernel on small grids, a memset on large ones and where J is
# off the 16-byte grid (an odd number of nodes)
@pytest.mark.parametrize("nx,nz,zeroing", [(64, 255, 1), (63, 256, 0), (2048, 1599, 0)])
def test_reported_launches(nx, nz, zeroing):
    import paper_1011_0917_gb300 as P
    sim = P.Simulation(dim=2, nx=nx, nz=nz, dx=1.0, dz=0.1, filter_passes=2, slots_per_cell=1.0)
    P.pic_profile_read(sim.ctx)

    def launches(mask):
        sim.step_phases(mask)
        return P.pic_profile_read(sim.ctx)[2]

    assert launches(1) == zeroing
    assert launches(32) == 1
    # zeroed, filtered and updated in one call: the raw current lies in scratch, which is aligned
    assert launches(1 | 16 | 32) == 2 + (nx < 1000)
    sim.close()
