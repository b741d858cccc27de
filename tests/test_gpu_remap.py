"""Lattices on the resident steps whose region map changes: steps, on whatever takes them, keep the
bits of the layout that lb_info names, from the first map to the last, also where a map in
between has no resident plan."""
import numpy as np
import pytest

from lbinputs import band_map, couette

pytestmark = pytest.mark.gpu


def _patch(nx, ny, row, cols):
    m = band_map(nx, ny, 3)
    m[row, cols] = 1
    return m


@pytest.mark.parametrize("store", ["f32_dev", "f32", "f64", "bf16_dev"])
@pytest.mark.parametrize("nx,ny", [(136, 16), (160, 24)])
def test_maps_with_and_without_a_resident_plan(nx, ny, store):
    import paper_1007_4895_gb300 as lb

    def make(**kw):
        w = couette(nx=nx, ny=ny, rows=3)
        x, y = 2 * np.pi * np.arange(nx)[None, :] / nx, np.pi * np.arange(ny)[:, None] / ny
        w.init = (1.0 + 0.02 * np.sin(x) * np.cos(y), 0.03 * np.cos(x) * np.sin(y), 0.02 * np.sin(x) * np.cos(2 * y))
        w.cfl = 0.38
        return lb.Lattice.from_workload(w, store=store, **kw)
    a = make()
    named = a.info()["variant"]
    if named != (9 if store in ("f32", "f32_dev") else 0):
        pytest.skip("the layouts were faster here")
    b = make(variant=named)
    # rows of one set, rows that change set along x (no resident plan), and back
    for m in (None, band_map(nx, ny, 4, 2), _patch(nx, ny, ny // 2, slice(0, 128)), _patch(nx, ny, ny // 2 - 1, slice(128, None)),
              band_map(nx, ny, 3), np.ones((ny, nx), np.uint8), band_map(nx, ny, 2)):
        for lat in (a, b):
            if m is not None:
                lat.set_region_map(m)
            lat.step(9)
        assert a.info()["variant"] == named
        eff = b.effective_map()
        for s in (0, 1):
            assert np.array_equal(a.populations(s)[:, eff == s], b.populations(s)[:, eff == s]), s
    a.close()
    b.close()
