"""Mini-batch training on the cluster kernel (lb_mlp_train) against FP64 training by the
oracle's gradient and Adam step on the same shuffled batches, at batch sizes that leave
blocks without samples, end inside a tile, or take several tiles per block, and at sample
counts whose last batch is short."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


def _mt64(seed):
    """The 64-bit Mersenne twister (Matsumoto & Nishimura), which shuffles the samples."""
    s, m = [seed], 2 ** 64 - 1
    for i in range(1, 312):
        s.append((6364136223846793005 * (s[-1] ^ (s[-1] >> 62)) + i) & m)
    while True:
        for i in range(312):
            x = (s[i] & 0xFFFFFFFF80000000) | (s[(i + 1) % 312] & 0x7FFFFFFF)
            s[i] = s[(i + 156) % 312] ^ (x >> 1) ^ (0xB5026F5AA96619E9 if x & 1 else 0)
        for x in s:
            x ^= (x >> 29) & 0x5555555555555555
            x ^= (x << 17) & 0x71D67FFFEDA60000
            x ^= (x << 37) & 0xFFF7EEE000000000
            yield x ^ (x >> 43)


@pytest.mark.parametrize("n,batch,epochs", [(5, 1, 1), (300, 7, 1), (1000, 64, 2), (999, 200, 2), (4099, 256, 1),
                                            (5000, 257, 1), (9000, 2900, 2), (700, 4096, 3)])
def test_training_follows_the_oracle(n, batch, epochs):
    """The oracle's move from the start and the kernel's: FP32 gradients are off by about
    1e-6 of their largest component, and Adam turns a component's relative error into the
    same relative error of its step, at most a full step (lr) where the gradient is within
    rounding of zero; those are few. Over the vector the moves agree to 1e-3 of their norm,
    while a lost sample, a wrong order or a wrong step number moves them by O(1) of it."""
    import torch
    import paper_1007_4895_gb300 as lb
    rng = np.random.default_rng(n + batch)
    xn = rng.standard_normal((8, n)).astype(np.float32)
    y = ((xn[0] * xn[1] + 0.3 * xn[6]) > 0.1).astype(np.float32)
    theta = omlp.init_params(batch).astype(np.float32)
    m = lb.MLP(theta, np.concatenate([np.zeros(8), np.ones(8)]).astype(np.float32))
    last = m.train(torch.tensor(xn, device="cuda"), torch.tensor(y, device="cuda"), epochs=epochs, batch=batch, seed=77)
    th = theta.astype(np.float64)
    mo, vo, t = np.zeros_like(th), np.zeros_like(th), 0
    perm, draw, x64 = list(range(n)), _mt64(77), xn.T.astype(np.float64)
    for _ in range(epochs):
        for k in range(n - 1, 0, -1):
            r = next(draw) % (k + 1)
            perm[k], perm[r] = perm[r], perm[k]
        total = 0.0
        for s in range(0, n, batch):
            i = perm[s:s + batch]
            total += omlp.loss(th, x64[i], y[i]) * len(i)
            t += 1
            th, mo, vo = omlp.adam_step(th, mo, vo, omlp.grad(th, x64[i], y[i]), t)
    move, ref = m.params().astype(np.float64) - theta, th - theta
    assert np.linalg.norm(move - ref) <= 1e-3 * np.linalg.norm(ref)
    assert abs(last - total / n) <= 1e-4 * abs(total / n)
