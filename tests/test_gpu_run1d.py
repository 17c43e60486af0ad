"""A 1D run's blocks write into one another's shared memory: no write may come
before every block of the cluster has started, and none after one has left.
That order cannot be made to fail at will on a GPU (a block starts early almost
always), so it is read from the kernel's source; short runs on an idle GPU,
where the start of the blocks and the first exchange lie closest together, are
compared with stepping bit for bit."""
import os
import re

import numpy as np
import pytest

import crkdg_inputs as inp
from tests.pairing import make_pair_1d, to_planes

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_first_remote_write_follows_a_cluster_barrier():
    src = open(os.path.join(ROOT, "paper_2307_06471_gb300", "csrc", "step1d.cuh")).read()
    body = re.sub(r"//[^\n]*", "", src[src.index("step1d_kernel("):])
    arrive, wait = body.index("cluster.barrier_arrive()"), body.index("cluster.barrier_wait()")
    write, sync = body.index("map_shared_rank"), body.index("cluster.sync()")
    assert arrive < wait < write < sync


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("nx", [31, 60, 91, 240, 241, 500, 960])
def test_short_runs_on_an_idle_gpu(nx, prec):
    import torch
    for physics, per in (("advection", True), ("euler", True), ("euler", False)):
        bcs = (("periodic",), ("periodic",)) if per else (("outflow",), ("outflow",))
        gs, _ = make_pair_1d(nx, (0, 1), 2, physics, "ssprk3", bcs, prec)
        u = to_planes(inp.random_modal_state_1d(nx, 2, 3 if physics == "euler" else 1, seed=nx))
        dt = 0.02 / nx
        for n in (2, 3):
            gs.set_state(u, 0.0)
            for _ in range(n):
                gs.step(dt)
            want = gs.get_state()
            for _ in range(20):
                gs.set_state(u, 0.0)
                torch.cuda.synchronize()
                gs.run_fixed(n, dt)
                assert np.array_equal(gs.get_state(), want), (physics, n)
        gs.close()
