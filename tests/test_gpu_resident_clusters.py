"""The resident steps on a given number of blocks, one to sixteen: bands of rows down to two,
halo rows, wall rows and views of other blocks, periodic y from the last block to the first,
several rounds a step. Each has the bits of one launch per step."""
import numpy as np
import pytest

from lbinputs import couette
from test_gpu_resident import CASES, _stripes, _waves

pytestmark = pytest.mark.gpu

ALL = dict(CASES)
for _c in (2, 4, 8, 16):
    ALL[f"two_rows_a_block_{2 * _c}"] = lambda c=_c: couette(nx=8, ny=2 * c, rows=max(2, c // 3))
    ALL[f"periodic_rows_{2 * _c}"] = lambda c=_c: _stripes(12, 2 * c)
ALL["several_rounds_16x330"] = lambda: couette(nx=16, ny=330, rows=30)
ALL["several_rounds_64x140"] = lambda: couette(nx=64, ny=140, rows=14)


@pytest.mark.parametrize("cluster", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("store,rounding", [("f64", "nearest"), ("f32", "nearest"), ("f32_dev", "nearest"), ("f16_dev", "nearest"),
                                            ("bf16_dev", "stochastic")])
def test_every_cluster_size(store, rounding, cluster):
    import paper_1007_4895_gb300 as lb
    ran = 0
    for case, make in ALL.items():
        a = lb.Lattice.from_workload(_waves(make()), store=store, rounding=rounding)
        if lb._lib.lbi_resident_cluster(a.ctx, cluster) == cluster:
            ran += 1
            b = lb.Lattice.from_workload(_waves(make()), store=store, rounding=rounding,
                                         variant=9 if store in ("f32", "f32_dev") else 0)
            for n in (1, 2, 41, 2):
                a.step(n)
                b.step(n)
                for s in (0, 1):
                    assert np.array_equal(a.populations(s), b.populations(s), equal_nan=True), (case, n, s)
            assert lb._lib.lbi_resident_cluster(a.ctx, 0) == cluster
            b.close()
        a.close()
    assert ran >= 8
