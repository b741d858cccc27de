"""Resident steps whose plan is as large as a block's shared memory: the batch runs and has the
bits of its lattice alone. The sizes came to exactly 227 KB when the plans took the kernel's
static word for theirs too."""
import numpy as np
import pytest

from lbinputs import couette

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,rows,store", [(8, 148, 2, "f64"), (16, 118, 10, "f32"), (16, 262, 10, "f16_dev"),
                                              (16, 262, 10, "bf16_dev")])
def test_a_plan_that_fills_the_block(nx, ny, rows, store):
    import paper_1007_4895_gb300 as lb
    b = lb.Batch([couette(nx=nx, ny=ny, rows=rows)], store=store)
    b.step(3)
    b.sync()
    alone = lb.Lattice.from_workload(couette(nx=nx, ny=ny, rows=rows), store=store, variant=0 if store == "f64" else 9)
    alone.step(3)
    for s in (0, 1):
        assert np.array_equal(b.lattice(0).populations(s), alone.populations(s)), s
    b.close()
    alone.close()
