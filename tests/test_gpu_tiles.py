"""Layout 10 on tiles streamed by the tensor memory accelerator (lattices whose two levels
fit L2) and on rows through the per-thread ring (larger ones), against layout 9: the same
bits, at widths that end on a tile, inside one, inside a quad, at heights that leave units of
one to seven rows, with walls, pressure columns, periodic columns and rows, shadows, mode-A
interface rows and a per-column reference density."""
import numpy as np
import pytest

from lbinputs import Workload, couette, long_channel, long_channel_density, poiseuille

pytestmark = pytest.mark.gpu


def _stripes(nx, ny):
    m = np.zeros((ny, nx), np.uint8)
    m[[0, 1, 2, 9, 17, 18]] = 1
    m[5:7, :nx // 2] = 1          # sets that change along x
    side = {"kind": "periodic"}
    return Workload(name="stripes", nx=nx, ny=ny, region_map=m, kn_ref=0.2, gy=0.1, walls={"bottom": side, "top": side})


CASES = {
    "force_256x40": lambda: poiseuille(nx=256, ny=40, rows=6, g_lat=1e-4),
    "force_130x23": lambda: poiseuille(nx=130, ny=23, rows=3, g_lat=1e-4),
    "couette_5x9": lambda: couette(nx=5, ny=9, rows=2),
    "couette_127x30_16": lambda: couette(nx=127, ny=30, rows=5, sets=(9, 16)),
    "mode_a_200x48": lambda: couette(nx=200, ny=48, rows=9, iface="paper"),
    "stripes_256x24": lambda: _stripes(256, 24),
    "stripes_301x26": lambda: _stripes(301, 26),
    "long_384x41": lambda: long_channel(nx=384, ny=41),
    "long_300x37": lambda: long_channel(nx=300, ny=37),
    "long_640x64_all_high": lambda: _all_high(640, 64),
}


def _all_high(nx, ny):
    w = long_channel(nx=nx, ny=ny, cfl=0.38)
    w.region_map = np.ones((ny, nx), np.uint8)
    return w


def _same(w, store, steps, **kw):
    import paper_1007_4895_gb300 as lb
    a = lb.Lattice.from_workload(w, store=store, variant=10, **kw)
    b = lb.Lattice.from_workload(w, store=store, variant=9, **kw)
    assert a.info()["variant"] == 10 and b.info()["variant"] == 9
    for n in steps:
        a.step(n)
        b.step(n)
        eff = a.effective_map()
        for s in (0, 1):
            assert np.array_equal(a.populations(s)[:, eff == s], b.populations(s)[:, eff == s]), (n, s)
    assert a.sync() == 0   # no wait ran out
    a.close()
    b.close()


@pytest.mark.parametrize("store", ["f32", "f32_dev", "f16_dev", "bf16_dev"])
@pytest.mark.parametrize("case", list(CASES))
def test_tiles_equal_the_ring_layout(case, store):
    w = CASES[case]()
    if w.init is None:
        x = 2 * np.pi * np.arange(w.nx)[None, :] / w.nx
        y = np.pi * np.arange(w.ny)[:, None] / w.ny
        w.init = (1.0 + 0.02 * np.sin(x) * np.cos(y), 0.03 * np.cos(x) * np.sin(y), 0.02 * np.sin(x) * np.cos(2 * y))
        w.cfl = 0.38
    _same(w, store, (7, 8))


def test_tiles_with_a_per_column_reference():
    w = long_channel(nx=500, ny=33)
    _same(w, "f32_dev", (5, 4), rho0_col=long_channel_density(w.nx, 2.0, 1.0))


def test_lattice_beyond_l2_equals_the_ring_layout():
    _same(long_channel(nx=8192, ny=128), "f32_dev", (3,))
