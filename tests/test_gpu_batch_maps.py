"""A member of a batch that gets another region map (by a call, or by a checkpoint): the batch
steps it as the same lattice alone, whichever kernel the batch runs on before and after."""
import numpy as np
import pytest

from lbinputs import band_map, couette, poiseuille

pytestmark = pytest.mark.gpu


def _waves(w):
    x = 2 * np.pi * np.arange(w.nx)[None, :] / w.nx
    y = np.pi * np.arange(w.ny)[:, None] / w.ny
    w.init = (1.0 + 0.02 * np.sin(x + 0.3) * np.cos(y), 0.03 * np.cos(x) * np.sin(2 * y) + 0 * x,
              0.02 * np.sin(2 * x) * np.cos(y))
    w.cfl = 0.38
    return w


def _workloads(nx, heights):
    return [_waves(couette(nx=nx, ny=ny, rows=max(2, ny // 7)) if k % 2 else
                   poiseuille(nx=nx, ny=ny, rows=max(2, ny // 6), kn=0.1 + 0.1 * k, g_lat=1e-3))
            for k, ny in enumerate(heights)]


def _patch(nx, ny):
    """Walls, and one tile of the core: a map that changes along x where nx > 128."""
    m = band_map(nx, ny, 3)
    m[ny // 2, :128] = 1
    return m


def _same(b, alone, what):
    for i, lat in enumerate(alone):
        if lat is None:
            continue
        eff = lat.effective_map()
        assert np.array_equal(b.lattice(i).effective_map(), eff), (what, i)
        for s in (0, 1):
            got, ref = b.lattice(i).populations(s), lat.populations(s)
            assert np.array_equal(got[:, eff == s], ref[:, eff == s]), (what, i, s)


# resident throughout; to a map whose rows no longer fit a block, and back; rows that change set
# along x; never resident (too tall, or 16-bit and wider than a tile)
@pytest.mark.parametrize("nx,heights,store", [
    (8, (16, 33, 70, 21), "f64"), (8, (16, 33, 70, 21), "f32_dev"), (8, (16, 33, 70, 21), "bf16_dev"),
    (13, (12, 40), "f32"), (8, (16, 200, 30), "f64"), (8, (16, 250, 30), "f32_dev"), (8, (16, 250, 30), "f32"),
    (140, (12, 10), "f64"), (96, (200, 24), "f32_dev"), (96, (220, 24), "bf16_dev"), (140, (30, 20), "f16_dev")])
def test_member_with_another_map(nx, heights, store):
    import paper_1007_4895_gb300 as lb
    b = lb.Batch(_workloads(nx, heights), store=store)
    ring = store != "f64" and nx <= 128
    alone = [lb.Lattice.from_workload(w, store=store, variant=9 if ring else 0) for w in _workloads(nx, heights)]

    def step(n, what):
        b.step(n)
        for lat in alone:
            lat.step(n)
        _same(b, alone, what)

    def remap(i, m):
        for lat in (b.lattice(i), alone[i]):
            lat.set_region_map(m)
    step(5, "start")
    ny = heights[1]
    remap(1, band_map(nx, ny, 2, 5))
    step(4, "bands")
    remap(0, _patch(nx, heights[0]))
    remap(1, np.ones((ny, nx), np.uint8))
    step(3, "patch and all high")
    remap(1, np.zeros((ny, nx), np.uint8))
    remap(0, band_map(nx, heights[0], 3))
    step(6, "back")
    b.graph(4, replays=2)
    b.step_each(3)
    for lat in alone:
        lat.step(11)
    _same(b, alone, "graph and single steps")
    b.close()


@pytest.mark.parametrize("store", ["f64", "f32_dev"])
def test_member_loaded_from_a_checkpoint_of_another_map(store, tmp_path):
    import paper_1007_4895_gb300 as lb
    ws = _workloads(8, (24, 40))
    src = lb.Lattice.from_workload(_workloads(8, (24, 40))[1], store=store, variant=0 if store == "f64" else 9)
    src.step(3)
    src.set_region_map(band_map(8, 40, 9, 4))
    src.step(2)
    src.save(str(tmp_path / "c"))
    b = lb.Batch(ws, store=store)
    b.step(4)
    b.lattice(1).load(str(tmp_path / "c"))
    b.step(7)
    src.step(7)
    _same(b, [None, src], "loaded")
    b.close()
