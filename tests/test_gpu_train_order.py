"""Training over several epochs takes its samples in the seeded order of each
epoch: the order is rewritten on the host while the last epoch's minibatches run
(many, and slow against a shuffle), so the copy to the GPU must have read it.

Reference: the same minibatches one by one through loss_grad and Adam in numpy
FP32 (which differ in the rounding of a division and a square root: a few 1e-7 of
each update, of which there are 192, in parameters of order 0.1); the band is
checked against what another order gives."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
N, BATCH, EPOCHS, LR = 2048, 32, 3, 1e-3
M64 = (1 << 64) - 1


def splitmix(s):
    s = (s + 0x9E3779B97F4A7C15) & M64
    z = s
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return s, z ^ (z >> 31)


def orders(n, epochs, seed):
    perm, s = list(range(n)), seed
    for _ in range(epochs):
        for i in range(n - 1, 0, -1):
            s, z = splitmix(s)
            j = z % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        yield list(perm)


def by_hand(net, p0, X, y, seed):
    import torch
    f = np.float32
    p, m, v = p0.copy(), np.zeros_like(p0), np.zeros_like(p0)
    t = 0
    for perm in orders(N, EPOCHS, seed):
        for b in range(0, N, BATCH):
            idx = torch.tensor(perm[b:b + BATCH], device="cuda")
            Xb, yb = X[idx].contiguous(), y[idx].contiguous()
            torch.cuda.synchronize()
            net.set_params(p)
            _, g = net.loss_grad(Xb.data_ptr(), yb.data_ptr(), len(idx))
            t += 1
            c1, c2 = f(1.0 - float(f(0.9)) ** t), f(1.0 - float(f(0.999)) ** t)
            m = f(0.9) * m + (f(1) - f(0.9)) * g
            v = f(0.999) * v + (f(1) - f(0.999)) * g * g
            p = (p - f(LR) * (m / c1) / (np.sqrt(v / c2) + f(1e-8))).astype(f)
    return p


def test_order_of_every_epoch():
    import torch
    from paper_2307_06471_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(4)
    X = torch.randn(N, 40, generator=g, device="cuda")
    y = (X[:, 0] + X[:, 1] * X[:, 2] > 0.5).float()
    torch.cuda.synchronize()
    net = B.MLP(seed=6)
    p0 = net.get_params()
    want, other = by_hand(net, p0, X, y, 11), by_hand(net, p0, X, y, 12)
    moved = np.linalg.norm(want - p0)
    band = 0.02 * moved
    assert np.linalg.norm(want - other) > 5 * band
    for _ in range(5):
        net.set_params(p0)
        net.train(X.data_ptr(), y.data_ptr(), N, EPOCHS, BATCH, LR, seed=11)
        assert np.linalg.norm(net.get_params() - want) < band
    net.close()
