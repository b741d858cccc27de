"""Layout 10 on tiles with units that leave most of a block's warps without a row: those warps
pass the unit's stages over, and release a stage only after every lane has seen it full. Single
rows of either set, over many steps: the bits of layout 9, and no wait runs out."""
import numpy as np
import pytest

from lbinputs import Workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", ["f32_dev", "bf16_dev"])
@pytest.mark.parametrize("nx,ny,rows", [(640, 24, (0, 1, 5, 9, 13, 17, 22, 23)), (384, 16, (0, 1, 8, 14, 15)),
                                        (131, 12, (0, 1, 4, 6, 10, 11))])
def test_units_of_few_rows(nx, ny, rows, store):
    import paper_1007_4895_gb300 as lb
    m = np.zeros((ny, nx), np.uint8)
    m[list(rows)] = 1
    x, y = 2 * np.pi * np.arange(nx)[None, :] / nx, np.pi * np.arange(ny)[:, None] / ny
    wall = {"kind": "diffuse"}
    w = Workload(name="single rows", nx=nx, ny=ny, region_map=m, kn_ref=0.3, cfl=0.38,
                 walls={"bottom": {**wall, "ux": -0.05}, "top": {**wall, "ux": 0.05}})
    w.init = (1.0 + 0.02 * np.sin(x) * np.cos(y), 0.03 * np.cos(x) * np.sin(y), 0.02 * np.sin(x) * np.cos(2 * y))
    a = lb.Lattice.from_workload(w, store=store, variant=10)
    b = lb.Lattice.from_workload(w, store=store, variant=9)
    assert a.info()["variant"] == 10 and b.info()["variant"] == 9
    a.step(300)
    b.step(300)
    eff = a.effective_map()
    for s in (0, 1):
        assert np.array_equal(a.populations(s)[:, eff == s], b.populations(s)[:, eff == s]), s
    assert a.sync() == 0
    a.close()
    b.close()
