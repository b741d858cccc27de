"""Bundles of the resident steps where lattices cannot share a block: batches of several widths
(a bundle has one), of several time steps (equal population constants), and in FP64, in one launch
and over several. Every lattice has the bits of the same lattice alone."""
import numpy as np
import pytest

from lbinputs import couette, poiseuille

pytestmark = pytest.mark.gpu


def _workloads():
    out = []
    for k, (nx, ny) in enumerate([(8, 20), (13, 20), (8, 33), (16, 12), (5, 9), (13, 41), (4, 64), (8, 20), (32, 16), (7, 25)]):
        w = poiseuille(nx=nx, ny=ny, rows=2 + k % 3, kn=0.1 + 0.05 * k, g_lat=1e-3) if k % 2 else couette(nx=nx, ny=ny, rows=2 + k % 2)
        x, y = 2 * np.pi * np.arange(nx)[None, :] / nx, np.pi * np.arange(ny)[:, None] / ny
        w.init = (1.0 + 0.02 * np.sin(x) * np.cos(y), 0.03 * np.cos(x) * np.sin(y), 0.02 * np.sin(x) * np.cos(2 * y))
        w.cfl = 0.38 if k < 7 else 0.3
        out.append(w)
    return out


@pytest.mark.parametrize("store", ["f64", "f32", "f32_dev", "f16_dev", "bf16_dev"])
def test_mixed_bundles_equal_lattices_alone(store):
    import paper_1007_4895_gb300 as lb
    b = lb.Batch(_workloads(), store=store)
    b.step(30)
    b.step(17)
    for i, w in enumerate(_workloads()):
        alone = lb.Lattice.from_workload(w, store=store, variant=0 if store == "f64" else 9)
        alone.step(47)
        for s in (0, 1):
            assert np.array_equal(b.lattice(i).populations(s), alone.populations(s)), (i, s)
        assert b.lattice(i).info()["step"] == 47
        alone.close()
    b.close()
