"""1D runs on few cells: stepping and runs (of one block, of a cluster) do the same
operations in the same order, bit for bit, for every degree; and a step of a
small FP32 Euler run, whose arithmetic takes a microsecond, does not spend more
than that on FP64 conversions of the scheme's constants (3.3 us a step; 2.3 us
when the run went through global memory)."""
import numpy as np
import pytest

import crkdg_inputs as inp
from tests.pairing import make_pair_1d, to_planes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("k", [0, 1, 2, 3])
@pytest.mark.parametrize("nx", [7, 31, 60, 61, 91, 240, 241, 500, 960])
def test_runs_equal_steps(nx, k, prec):
    import torch
    for physics, per in (("advection", True), ("euler", True), ("euler", False)):
        bcs = (("periodic",), ("periodic",)) if per else (("outflow",), ("outflow",))
        gs, _ = make_pair_1d(nx, (0, 1), k, physics, "ssprk3", bcs, prec)
        u = to_planes(inp.random_modal_state_1d(nx, k, 3 if physics == "euler" else 1, seed=nx))
        dt = 0.02 / nx
        for n in (2, 3):
            gs.set_state(u, 0.0)
            for _ in range(n):
                gs.step(dt)
            want = gs.get_state()
            for _ in range(5):
                gs.set_state(u, 0.0)
                torch.cuda.synchronize()
                gs.run_fixed(n, dt)
                assert np.array_equal(gs.get_state(), want), (physics, n)
        gs.close()


def step_ms(k, nx, precision):
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    stream = torch.cuda.Stream()
    mesh = B.make_mesh(1, nx, 1, (0.0, 1.0, 0.0, 1.0), [B.BC_PERIODIC] * 4)
    s = B.Solver(mesh, k, B.BASIS_P, T.SSPRK3, B.EULER, precision, stream=stream.cuda_stream)
    s.set_state(to_planes(inp.random_modal_state_1d(nx, k, 3, seed=nx)))
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = []
    with torch.cuda.stream(stream):
        for _ in range(7):
            e0.record(stream)
            s.run_fixed(400, 1e-5 / nx)
            e1.record(stream)
            stream.synchronize()
            times.append(e0.elapsed_time(e1) / 400)
    s.close()
    return sorted(times)[3]


# part of the FP64 run's step: 0.125, 0.082, 0.066 and 0.20 measured; 0.30, 0.18, 0.14
# and 0.32 with the conversions
@pytest.mark.parametrize("k,nx,part", [(0, 45, 0.2), (1, 45, 0.13), (2, 45, 0.1), (0, 160, 0.26)])
def test_time_of_a_small_euler_step(k, nx, part):
    from paper_2307_06471_gb300 import binding as B
    assert step_ms(k, nx, B.F32) < part * step_ms(k, nx, B.F64)
