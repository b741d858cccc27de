"""One host thread per lattice, each on its own stream, stepping at the same time while a third
creates lattices: every call succeeds, and every lattice has the bits of the same run alone."""
import threading

import numpy as np
import pytest

from lbinputs import couette

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", ["f32_dev", "f64"])
def test_threads_step_and_create_lattices(store):
    import torch
    import paper_1007_4895_gb300 as lb
    sizes = [(8, 24), (16, 90), (8, 60)]
    calls = 800

    def make(size):
        return lb.Lattice.from_workload(couette(nx=size[0], ny=size[1], rows=4), store=store, stream=torch.cuda.Stream(),
                                        torch_allocator=False)
    want = []
    for size in sizes:
        lat = make(size)
        lat.step(calls)
        want.append([lat.populations(s) for s in (0, 1)])
        lat.close()
    lats, errors, done = [make(size) for size in sizes], [], threading.Event()

    def step(lat):
        try:
            for _ in range(calls):
                lat.step(1)
            lat.sync()
        except Exception as e:   # noqa: BLE001
            errors.append(repr(e))

    def create():
        k = 0
        try:
            while not done.is_set():
                lat = lb.Lattice.from_workload(couette(nx=12, ny=20 + k % 50, rows=3), store=store, stream=torch.cuda.Stream(),
                                               torch_allocator=False)
                lat.step(2)
                lat.sync()
                lat.close()
                k += 1
        except Exception as e:   # noqa: BLE001
            errors.append("create: " + repr(e))
    threads = [threading.Thread(target=step, args=(lat,)) for lat in lats]
    maker = threading.Thread(target=create)
    maker.start()
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    done.set()
    maker.join()
    assert not errors, errors[:3]
    for lat, ref in zip(lats, want):
        for s in (0, 1):
            assert np.array_equal(lat.populations(s), ref[s])
        lat.close()
