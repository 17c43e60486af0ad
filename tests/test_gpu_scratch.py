"""Scratch that launches and recorded graphs point to: calls between two runs of
a graph must not move it, or the graph must be recorded again."""
import numpy as np
import pytest

import crkdg_inputs as inp
from tests.pairing import to_planes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_graph_of_modal_steps_outlives_rkdg_steps(prec):
    """A linear context whose quadrature step (crkdg_rkdg_step's) has far more
    segments, and reduction slots, than its modal step: graph replays before and
    after an RKDG step, a dt and the totals equal steps that are not captured."""
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    nx, ny = 331, 1200
    mesh = B.make_mesh(2, nx, ny, (0.0, 1.0, 0.0, 3.6), [B.BC_PERIODIC] * 4)
    u = to_planes(inp.random_modal_state(ny, nx, 1, "P", "advection", seed=3))
    stream = torch.cuda.Stream()
    out = []
    for capture in (False, True):
        s = B.Solver(mesh, 1, B.BASIS_P, T.HEUN2, B.ADVECTION, B.F32 if prec == "f32" else B.F64, beta=(1.0, 0.5),
                     stream=stream.cuda_stream)
        s.set_launch(1, 0)
        s.set_state(u, 0.0)
        s.advance(4, 0.1, 10.0, capture=capture)
        s.rkdg_step(1e-5, 2)
        dt = s.cfl_dt(0.1)
        tot = s.conservation()
        s.advance(4, 0.1, 10.0, capture=capture)
        s.rkdg_step(1e-5, 2)
        s.advance(4, 0.1, 10.0, capture=capture)
        out.append((s.get_state(), s.time(), dt, tuple(tot), s.step_count()))
        assert s.sync() == (0, 0)
        s.close()
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1:] == out[1][1:]
