"""Calls from several threads on one handle that share its kept workspace: the
read-back of a batch's problems, the loss and gradient of a network."""
import threading

import numpy as np
import pytest

import crkdg_inputs as inp
from tests.pairing import to_planes

pytestmark = pytest.mark.gpu


def in_threads(jobs):
    errors, gate = [], threading.Barrier(len(jobs))

    def body(job):
        try:
            gate.wait()
            job()
        except BaseException as e:   # noqa: B902
            errors.append(e)
    ts = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if errors:
        raise errors[0]


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("limited", [False, True])
def test_batch_read_back(prec, limited):
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    sizes = [(20, 30), (64, 33), (150, 140), (200, 256)]
    stream = torch.cuda.Stream()
    make = lambda: B.Batch([(nx, ny, (0.0, 1.0, 0.0, 1.0)) for nx, ny in sizes], 2, B.BASIS_P, T.SSPRK3,  # noqa: E731
                           B.F64 if prec == "f64" else B.F32, stream=stream.cuda_stream)
    states = [to_planes(inp.random_modal_state(ny, nx, 2, "P", "euler", seed=i, amp=0.3)) for i, (nx, ny) in enumerate(sizes)]

    def fill(b):
        for i, u in enumerate(states):
            b.set_state(i, u)
        if limited:
            b.limit(1.0)
        return b
    a = fill(make())
    want = [a.get_state(i) for i in range(len(sizes))]
    a.close()
    for _ in range(3):
        b = fill(make())

        def reads(first):
            for k in range(8):
                i = (first + k) % len(sizes)
                assert np.array_equal(b.get_state(i), want[i])
        in_threads([lambda i=i: reads(i) for i in range(4)])
        b.close()


def test_loss_and_gradient():
    import torch
    from paper_2307_06471_gb300 import binding as B
    X = torch.randn(30000, 40, device="cuda")
    y = (X[:, 0] > 0.5).float()
    torch.cuda.synchronize()
    sizes = [7, 500, 3000, 30000]
    net = B.MLP(seed=2)
    p = net.get_params()
    want = [net.loss_grad(X.data_ptr(), y.data_ptr(), n) for n in sizes]
    net.close()
    for _ in range(3):
        net = B.MLP(seed=2)
        assert np.array_equal(net.get_params(), p)

        def evals(first):
            for k in range(8):
                i = (first + k) % len(sizes)
                loss, g = net.loss_grad(X.data_ptr(), y.data_ptr(), sizes[i])
                assert loss == want[i][0] and np.array_equal(g, want[i][1])
        in_threads([lambda i=i: evals(i) for i in range(4)])
        net.close()
