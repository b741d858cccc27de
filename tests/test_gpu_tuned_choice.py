"""The resident steps and the layouts are compared by their times also where the layouts' come from
an earlier lattice of the same size and map."""
import pytest

from lbinputs import band_map, couette

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(160, 24), (136, 16)])
def test_a_known_layout_time_is_compared(nx, ny):
    import paper_1007_4895_gb300 as lb
    a = lb.Lattice.from_workload(couette(nx=nx, ny=ny, rows=3), store="f64")
    named = a.info()["variant"]
    a.close()
    if named == 0:   # layout 0, or the resident steps, which go by its name
        pytest.skip("layout 0 or the resident steps were faster here")
    # the walls differ (periodic y), the layouts' cache does not: the same layout, not the slower steps
    side = {"kind": "periodic"}
    w = couette(nx=nx, ny=ny, rows=3)
    b = lb.Lattice(nx, ny, band_map(nx, ny, 3), kn_ref=w.kn_ref, walls={"bottom": side, "top": side}, store="f64", cfl=w.cfl)
    assert b.info()["variant"] == named
    b.close()
