"""An allocator that refuses what the resident steps want on top of a lattice: the lattice is
created all the same and runs on the layouts, also where an earlier one of its kind took the
resident steps."""
import numpy as np
import pytest

from lbinputs import couette

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", ["f32_dev", "f64", "bf16_dev"])
def test_creation_without_memory_for_a_plan(store):
    import torch
    import paper_1007_4895_gb300 as lb
    w = couette(nx=8, ny=64, rows=4)
    first = lb.Lattice.from_workload(w, store=store)
    freed, refused = [], []

    def alloc(nbytes, user):
        if freed:   # the buffer of the initial state has been given back: what follows is the plan's
            refused.append(nbytes)
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes))

    def free(ptr, user):
        freed.append(ptr)
        torch.cuda.caching_allocator_delete(ptr)
    opts = lb.lb_opts()
    opts.store, opts.iface, opts.rho0, opts.variant = lb.STORES[store], lb.LB_IFACE_HERMITE, w.rho0, -1
    opts.stream = torch.cuda.current_stream().cuda_stream
    opts.alloc, opts.free = lb.ALLOC_FN(alloc), lb.FREE_FN(free)
    ctx = lb.lb_create(lb.lb_grid(w.nx, w.ny, 0.0, w.cfl, 0.0), w.region_map, w.sets, lb.lb_kn(w.kn_ref, w.rho_ref, 0),
                       lb._walls(w.walls), opts)
    assert refused
    lb.lb_step(ctx, 20)
    first.step(20)
    out = torch.empty((3, w.ny, w.nx), dtype=torch.float64, device="cuda")
    lb.lb_moments(ctx, 0b111, out.data_ptr(), 1, 1)
    out = out.cpu().numpy()
    ref = first.moments()
    tol = {"f64": 1e-12, "f32_dev": 1e-6}.get(store, 2e-2)
    for k, name in enumerate(("rho", "ux", "uy")):
        assert np.abs(out[k] - ref[name]).max() <= tol
    lb.lb_destroy(ctx)
    first.close()
