"""Pressure channels whose last tile of 128 columns holds the boundary column alone, or a few: the
boundary column needs the node one step inwards of the same step, which is then another tile's.
Layout 10, on tiles and (a lattice beyond L2) on rows, against layout 9, whose pressure pass is a
launch of its own: the same bits, step after step."""
import numpy as np
import pytest

from lbinputs import long_channel, long_channel_density

pytestmark = pytest.mark.gpu


def _same(w, store, rounds, **kw):
    import paper_1007_4895_gb300 as lb
    a = lb.Lattice.from_workload(w, store=store, variant=10, **kw)
    b = lb.Lattice.from_workload(w, store=store, variant=9, **kw)
    assert a.info()["variant"] == 10 and b.info()["variant"] == 9
    for n in rounds:
        a.step(n)
        b.step(n)
        eff = a.effective_map()
        for s in (0, 1):
            assert np.array_equal(a.populations(s)[:, eff == s], b.populations(s)[:, eff == s]), (n, s)
    assert a.sync() == 0
    a.close()
    b.close()


@pytest.mark.parametrize("store", ["f32", "f32_dev", "f16_dev", "bf16_dev"])
@pytest.mark.parametrize("nx,ny", [(129, 33), (257, 41), (385, 24), (1153, 64), (130, 33), (131, 20), (384, 17)])
def test_last_tile_of_few_columns(nx, ny, store):
    _same(long_channel(nx=nx, ny=ny, cfl=0.38), store, (1, 1, 2, 7, 30, 60))


def test_last_tile_of_one_column_with_a_per_column_reference():
    w = long_channel(nx=641, ny=33, cfl=0.38)
    _same(w, "f32_dev", (1, 5, 4, 30), rho0_col=long_channel_density(w.nx, 2.0, 1.0))


def test_last_tile_of_one_column_beyond_l2():
    _same(long_channel(nx=8193, ny=128, cfl=0.38), "f32_dev", (1, 2, 9))
