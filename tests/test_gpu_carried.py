"""Moments carried by layout 10, summed once from an initialised or loaded state (a quad of
columns per thread): the next step has layout 9's bits, which sums its own, at widths that
end on each column of a quad, on a tile and inside one, for every storage and set."""
import numpy as np
import pytest

from lbinputs import couette, long_channel, long_channel_density

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", ["f32", "f32_dev", "f16_dev", "bf16_dev"])
@pytest.mark.parametrize("nx,ny,sets", [(5, 9, (9, 36)), (6, 11, (9, 16)), (7, 9, (9, 36)), (8, 33, (9, 36)),
                                        (127, 10, (9, 16)), (128, 9, (9, 36)), (259, 21, (9, 36)), ("col", 17, (9, 36))])
def test_first_step_after_init_and_load(nx, ny, sets, store):
    import paper_1007_4895_gb300 as lb
    kw = {}
    if nx == "col":
        if store == "f32":
            pytest.skip("a per-column reference needs a deviation format")
        w = long_channel(nx=390, ny=ny)
        kw["rho0_col"] = long_channel_density(w.nx, 2.0, 1.0)
    else:
        w = couette(nx=nx, ny=ny, rows=3, sets=sets)
        w.cfl = 0.38
        x, y = 2 * np.pi * np.arange(nx)[None, :] / nx, np.pi * np.arange(ny)[:, None] / ny
        w.init = (1.0 + 0.02 * np.sin(x) * np.cos(y), 0.03 * np.cos(x) * np.sin(y), 0.02 * np.sin(x) * np.cos(2 * y))
    a = lb.Lattice.from_workload(w, store=store, variant=10, **kw)
    b = lb.Lattice.from_workload(w, store=store, variant=9, **kw)
    assert a.info()["variant"] == 10 and b.info()["variant"] == 9
    n = a.state_bytes()
    first, got, want = (np.zeros(n, np.uint8) for _ in range(3))
    lb.lb_state_store(a.ctx, first.ctypes.data, n)
    for _ in range(2):
        for lat, out in ((a, got), (b, want)):
            lat.step(1)
            lb.lb_state_store(lat.ctx, out.ctypes.data, n)
            lat.sync()
        assert np.array_equal(got, want)
        for lat in (a, b):
            lb.lb_state_load(lat.ctx, first.ctypes.data, n)
    a.close()
    b.close()
