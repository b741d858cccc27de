"""Inference with one and with two tiles of 16 nodes per warp (few nodes and many): a node's p does
not depend on how many nodes are asked for, or on its place among them, up to the last, ragged
tile; a node with a non-finite feature has no p, and its neighbours keep theirs."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


def test_p_does_not_depend_on_the_count():
    import torch
    import paper_1007_4895_gb300 as lb
    net = lb.MLP(omlp.init_params(5).astype(np.float32), np.concatenate([np.zeros(8), np.ones(8)]).astype(np.float32))
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(8, 120001, device="cuda", generator=g)
    x[3, 7] = float("nan")
    x[0, 48641] = float("inf")

    def infer(lo, hi):
        out = torch.full((hi - lo + 3,), 7.0, device="cuda")
        net.infer(x[:, lo:hi].contiguous(), out[:hi - lo])
        assert bool((out[hi - lo:] == 7.0).all())
        return out[:hi - lo].cpu().numpy()
    want = infer(0, x.shape[1])
    assert np.isnan(want[[7, 48641]]).all() and np.isnan(want).sum() == 2
    # 48640 nodes fill the resident warps with a tile each: the last count with one per warp
    for lo, hi in ((0, 1), (0, 15), (3, 20), (5, 517), (0, 48640), (0, 48641), (17, 48690), (1, 60002), (9, 120001)):
        assert np.array_equal(infer(lo, hi), want[lo:hi], equal_nan=True), (lo, hi)
    net.close()
