"""Layout 10 is among the layouts that lb_create times for a per-column reference density in FP32
deviations, whatever the size; the choice is the fastest of them within the tuner's margin."""
import pytest

from lbinputs import long_channel, long_channel_density

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(512, 64), (8192, 128)])
def test_per_column_lattices_take_layout_10(nx, ny):
    """At these sizes layout 10 takes 45 and 78 us a step and the next best layout 50 and 94: beyond
    the margin of 3 %."""
    import paper_1007_4895_gb300 as lb
    lat = lb.Lattice.from_workload(long_channel(nx=nx, ny=ny), store="f32_dev", rho0_col=long_channel_density(nx, 2.0, 1.0))
    assert lat.info()["variant"] == 10
    lat.close()
