"""Several steps per launch with the state in shared memory (the steps of small lattices)
against one launch per step: the same bits as layout 9 for FP32 storage and as layout 0 for
FP64 and 16-bit storage, whatever the width, the band structure, the number of blocks the
rows are spread over, and the way the steps are grouped into calls."""
import numpy as np
import pytest

from lbinputs import Workload, band_map, couette, kramers, oscillatory_couette, poiseuille

pytestmark = pytest.mark.gpu


def _waves(w):
    x = 2 * np.pi * np.arange(w.nx)[None, :] / w.nx
    y = np.pi * np.arange(w.ny)[:, None] / w.ny
    w.init = (1.0 + 0.02 * np.sin(x + 0.3) * np.cos(y), 0.03 * np.cos(x) * np.sin(2 * y) + 0 * x,
              0.02 * np.sin(2 * x) * np.cos(y))
    w.cfl = 0.38
    return w


def _stripes(nx, ny):
    """High-order rows in stripes of several heights, one row thin among them, periodic y."""
    m = np.zeros((ny, nx), np.uint8)
    for j in (0, 1, 2, 7, 12, 13, 14, 15, 20):
        m[j % ny] = 1
    side = {"kind": "periodic"}
    return Workload(name="stripes", nx=nx, ny=ny, region_map=m, kn_ref=0.2, gx=0.1, walls={"bottom": side, "top": side})


CASES = {
    "couette_4x32": lambda: couette(nx=4, ny=32, rows=4),
    "couette_5x16": lambda: couette(nx=5, ny=16, rows=2),
    "force_6x9": lambda: poiseuille(nx=6, ny=9, rows=2, kn=0.3, g_lat=1e-3),
    "force_7x21": lambda: poiseuille(nx=7, ny=21, rows=3, g_lat=1e-3),
    "force_8x64": lambda: poiseuille(nx=8, ny=64, rows=10, g_lat=1e-4),
    "couette_31x40_16": lambda: couette(nx=31, ny=40, rows=6, sets=(9, 16)),
    "all_high_12x24": lambda: couette(nx=12, ny=24, rows=12),
    "all_low_9x20": lambda: _low(9, 20),
    "high_low_sets_swapped": lambda: couette(nx=8, ny=30, rows=4, sets=(36, 9)),
    "stripes_10x24": lambda: _stripes(10, 24),
    "force_64x33": lambda: poiseuille(nx=64, ny=33, rows=5, g_lat=1e-4),
    "kramers_38x31": lambda: kramers(ny=31, span=10.0, layer=3.0, nx=38),
    "oscillating_9x41": lambda: oscillatory_couette(nx=9, ny=41),
}


def _low(nx, ny):
    w = couette(nx=nx, ny=ny, rows=1)
    w.region_map = np.zeros((ny, nx), np.uint8)
    return w


@pytest.mark.parametrize("store,rounding", [("f64", "nearest"), ("f32", "nearest"), ("f32_dev", "nearest"),
                                            ("f16_dev", "nearest"), ("bf16_dev", "nearest"), ("f16_dev", "stochastic"),
                                            ("bf16_dev", "stochastic")])
@pytest.mark.parametrize("case", list(CASES))
def test_resident_steps_equal_single_launches(case, store, rounding):
    import paper_1007_4895_gb300 as lb
    pair = store in ("f32", "f32_dev")
    a = lb.Lattice.from_workload(_waves(CASES[case]()), store=store, rounding=rounding)
    b = lb.Lattice.from_workload(_waves(CASES[case]()), store=store, rounding=rounding, variant=9 if pair else 0)
    # what the steps below must have run on: the layout that stands for them
    assert a.info()["variant"] == (9 if pair else 0)
    for n in (1, 2, 70, 3):
        a.step(n)
        b.step(n)
        for s in (0, 1):
            # every node of the set, and the views beside the interface, which the next step reads
            assert np.array_equal(a.populations(s), b.populations(s), equal_nan=True), (n, s)
    ra, rb = a.reductions(), b.reductions()
    assert ra == rb and ra["step"] == 76


@pytest.mark.parametrize("store", ["f32_dev", "f64", "bf16_dev"])
def test_resident_steps_stop_for_reductions_and_map_changes(store):
    """In-step reductions at an interval, then a map change to other bands: the same as with
    one launch per step."""
    import paper_1007_4895_gb300 as lb
    out = []
    for variant in (-1, 9 if store == "f32_dev" else 0):
        lat = lb.Lattice.from_workload(_waves(poiseuille(nx=20, ny=40, rows=5, g_lat=1e-4)), store=store, variant=variant,
                                       reduce_every=7)
        lat.step(20)
        lat.set_region_map(band_map(20, 40, 9, 3))
        lat.step(11)
        # each node in its own set (what it left in the other set before the map changed is unspecified)
        eff = lat.effective_map()
        out.append((lat.reductions(), lat.populations(0)[:, eff == 0], lat.populations(1)[:, eff == 1], lat.info()["step"]))
        lat.close()
    (ra, a0, a1, na), (rb, b0, b1, nb) = out
    assert ra == rb and na == nb == 31
    assert np.array_equal(a0, b0) and np.array_equal(a1, b1)


@pytest.mark.parametrize("store", ["f32", "f32_dev", "f16_dev", "bf16_dev"])
def test_bundles_of_lattices_equal_lattices_alone(store):
    """A batch small enough for the resident steps, of heights from one unit to many, and
    one whose lattices are too large for it (the other batch kernel)."""
    import paper_1007_4895_gb300 as lb

    def ws(nx, hs):
        return [_waves(couette(nx=nx, ny=ny, rows=max(2, ny // 7)) if k % 2 else
                       poiseuille(nx=nx, ny=ny, rows=max(2, ny // 6), kn=0.05 + 0.1 * k, g_lat=1e-3))
                for k, ny in enumerate(hs)]
    for nx, hs in ((8, (16, 9, 33, 70, 120, 17, 40, 8)), (13, (12, 21, 30)), (96, (200, 24))):
        b = lb.Batch(ws(nx, hs), store=store)
        b.step(4)
        b.step(9)
        for i, w in enumerate(ws(nx, hs)):
            alone = lb.Lattice.from_workload(w, store=store, variant=9)
            alone.step(13)
            for s in (0, 1):
                assert np.array_equal(b.lattice(i).populations(s), alone.populations(s)), (nx, i, s)
