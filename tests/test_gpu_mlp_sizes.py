"""The indicator's training, inference and feature kernels where their tiles
end: samples around the 8 of a training tile, the 32 of an inference warp and
the one wave of blocks, cells around the 128 of a features block, and an X that
allows no 8-byte loads.  Bands: the parity tests' 1e-5 for FP32 gradients
(summation order) and FP32 features; inference is the same whatever the
alignment."""
import numpy as np
import pytest

import crkdg_inputs as inp
from oracle import mlp as omlp
from oracle.limiter import neighbour_averages, tvb_limit
from tests.pairing import make_pair_2d, to_planes

pytestmark = pytest.mark.gpu


def _net(seed):
    from paper_2307_06471_gb300 import binding as B
    P = omlp.init_params(np.random.default_rng(seed))
    vec = np.concatenate([np.concatenate([W.reshape(-1), b.reshape(-1)]) for W, b in zip(P["W"], P["b"])]).astype(np.float32)
    net = B.MLP(seed=1)
    net.set_params(vec)
    o, Q = 0, {"W": [], "b": []}
    for a, b in ((64, 40), (64, 64), (64, 64), (1, 64)):
        Q["W"].append(vec[o:o + a * b].astype(np.float64).reshape(a, b))
        Q["b"].append(vec[o + a * b:o + a * b + a].astype(np.float64))
        o += a * b + a
    return net, Q


@pytest.mark.parametrize("n", [1, 7, 8, 9, 2431, 2433, 5000])
def test_gradient_sizes(n):
    import torch
    rng = np.random.default_rng(n)
    net, P = _net(3)
    X = rng.normal(size=(n, 40)).astype(np.float32)
    y = (rng.uniform(size=n) < 0.4).astype(np.float32)
    Xd, yd = torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda")
    loss, g = net.loss_grad(Xd.data_ptr(), yd.data_ptr(), n, pos_weight=1.5)
    z, cache = omlp.forward(P, X.astype(np.float64))
    L, dz = omlp.bce_with_logits(z, y.astype(np.float64), pos_weight=1.5)
    G = omlp.backward(P, cache, dz)
    want = np.concatenate([np.concatenate([W.reshape(-1), b.reshape(-1)]) for W, b in zip(G["W"], G["b"])])
    assert loss == pytest.approx(L, rel=1e-5)
    assert np.linalg.norm(g - want) <= 1e-5 * np.linalg.norm(want)
    net.close()


def test_training_is_the_sum_of_its_minibatches():
    """One epoch over a ragged last minibatch: the mean of its losses is finite
    and near the first loss, and training twice from the same parameters gives
    the same parameters (deterministic)."""
    import torch
    rng = np.random.default_rng(2)
    net, _ = _net(4)
    p0 = net.get_params()
    X = torch.tensor(rng.normal(size=(1000, 40)).astype(np.float32), device="cuda")
    y = (X[:, 0] > 0.5).float()
    out = []
    for _ in range(2):
        net.set_params(p0)
        loss = net.train(X.data_ptr(), y.data_ptr(), 1000, 1, 300, 1e-3, seed=5)
        out.append((loss, net.get_params()))
    l0, _ = net.loss_grad(X.data_ptr(), y.data_ptr(), 1000)
    assert out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1])
    assert l0 < out[0][0] < 2.0 and not np.array_equal(out[0][1], p0)
    net.close()


@pytest.mark.parametrize("n", [1, 31, 32, 33, 129, 100001])
def test_inference_sizes_and_alignment(n):
    import torch
    net, P = _net(5)
    buf = torch.randn(n * 40 + 1, device="cuda")
    a, b = (torch.full((n + 1,), -7.0, device="cuda") for _ in range(2))
    x = buf[1:].reshape(n, 40)                     # 4 bytes past an aligned address
    xa = x.clone()
    net.predict(xa.data_ptr(), n, a.data_ptr())
    net.predict(x.data_ptr(), n, b.data_ptr())
    assert torch.equal(a, b) and a[n] == -7.0      # nothing past the samples is written
    z, _ = omlp.forward(P, xa.cpu().numpy().astype(np.float64))
    assert np.max(np.abs(a[:n].cpu().numpy() - z)) < 0.05 * max(1.0, np.max(np.abs(z)))
    net.close()


@pytest.mark.parametrize("per", [True, False])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 5), (127, 3), (128, 2), (129, 4)])
def test_features_sizes(nx, ny, per):
    import torch
    bcs = {s: ("periodic",) if per else ("reflect",) for s in "WESN"}
    gs, dg = make_pair_2d(nx, ny, (0, 1.5, 0, 1.0), 2, "P", "euler", "ssprk3", bcs, "f64")
    u = inp.random_modal_state(ny, nx, 2, "P", "euler", seed=nx + ny, amp=0.3)
    gs.set_state(to_planes(u), 0.0)
    X = torch.full((nx * ny + 1, 40), -7.0, device="cuda")
    y = torch.full((nx * ny + 1,), -7.0, device="cuda")
    gs.features(X.data_ptr(), y.data_ptr(), 20.0)
    want = omlp.features(u, neighbour_averages(dg, u[..., 0], 0.0), 20.0, max(dg.dx, dg.dy))
    got = X.cpu().numpy().astype(np.float64)
    assert np.max(np.abs(got[:-1, :36] - want[:, :36])) < 1e-5
    assert np.max(np.abs(got[:-1, 36:] - want[:, 36:])) < 2e-5
    _, flags = tvb_limit(dg, u, 20.0, 0.0)
    assert np.array_equal(y[:-1].cpu().numpy().reshape(ny, nx) > 0.5, flags)
    assert (X[-1] == -7.0).all() and y[-1] == -7.0
    gs.close()
