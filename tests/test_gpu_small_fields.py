"""Small calls cost about what their one chain of work takes: moment fields of a tiny FP64 lattice
against its reduction (the same populations read and summed once more: 42 us each), which two nodes
per thread made 1.8 times as long."""
import pytest

from lbinputs import couette

pytestmark = pytest.mark.gpu


def _us(f, n=50):
    import torch
    best = 1e9
    for _ in range(5):
        f()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(n):
            f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, 1e3 * a.elapsed_time(b) / n)
    return best


def test_fp64_fields_of_a_tiny_lattice():
    import torch
    import paper_1007_4895_gb300 as lb
    lat = lb.Lattice.from_workload(couette(nx=4, ny=32, rows=4), store="f64")
    lat.step(2)
    out = torch.empty((9, 32, 4), dtype=torch.float64, device="cuda")
    fields, reduction = _us(lambda: lat.moments_into(out)), _us(lambda: lat.reductions())
    lat.close()
    assert fields <= 1.35 * reduction, (fields, reduction)
