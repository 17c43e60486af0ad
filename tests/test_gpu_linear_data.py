"""Linear advection with sine data on its sides: the modal step (the default)
against the quadrature step over every inflow direction, sides of each kind and
ragged sizes, and against the oracle; and 1D runs, whose cells stay in registers
and cross warps through shared memory, against stepping and the oracle at sizes
around a warp's 30 cells and the 8 blocks of a run.  Bands: FP64 1e-13 of the
scale per step between the forms and 1e-12 to the oracle, FP32 2e-5 (the parity
tests')."""
import numpy as np
import pytest

import crkdg_inputs as inp
from oracle.dg1d import crkdg_step as step1d
from oracle.dg2d import crkdg_step as step2d
from tests.pairing import TAB_NAMES, from_planes, make_pair_1d, make_pair_2d, rel_err, to_planes

pytestmark = pytest.mark.gpu
SINE = ("sine", 0.8, 2.0, 1.5, 3.0, 0.3)
PROD = ("sine_prod", 0.7, 3.0, 0.5, 2.0, 0.25)
OUT, CONST, PER = ("outflow",), ("const", [0.4]), ("periodic",)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2307_06471_gb300 import build
    build.build()


@pytest.mark.parametrize("beta", [(1.0, 0.5), (-1.0, 0.5), (1.0, -0.5), (-0.7, -1.0), (1.0, 0.0), (0.0, -1.0)])
@pytest.mark.parametrize("sides", [(SINE, SINE, SINE, SINE), (PROD, OUT, PROD, OUT), (OUT, PROD, CONST, SINE),
                                   (PER, PER, SINE, PROD), (SINE, PROD, PER, PER)])
@pytest.mark.parametrize("nx,ny,k,basis,tab,prec", [(31, 17, 3, "Q", "rk4", "f64"), (1, 1, 2, "Q", "heun3", "f64"),
                                                    (62, 2, 2, "P", "midpoint", "f64"), (45, 33, 2, "Q", "ssprk3", "f32")])
def test_modal_step_with_data(nx, ny, k, basis, tab, prec, sides, beta):
    from paper_2307_06471_gb300 import binding as B
    bcs = dict(zip("WESN", sides))
    gs, dg = make_pair_2d(nx, ny, (-1, 1, -0.6, 1), k, basis, "advection", tab, bcs, prec, beta=beta)
    u = inp.random_modal_state(ny, nx, k, basis, "advection", seed=nx)
    dt = 0.05 / (abs(beta[0]) * nx / 2 + abs(beta[1]) * ny / 1.6)
    got = {}
    for form in (B.FORM_AUTO, B.FORM_QUADRATURE):
        gs.set_operator_form(form)
        gs.set_state(to_planes(u), 0.25)
        for _ in range(3):
            gs.step(dt)
        got[form] = from_planes(gs.get_state())
    want, t = u, 0.25
    for _ in range(3):
        want = step2d(dg, want, t, dt, TAB_NAMES[tab])
        t += dt
    scale = np.max(np.abs(want))
    assert np.max(np.abs(got[B.FORM_AUTO] - got[B.FORM_QUADRATURE])) <= (3e-13 if prec == "f64" else 2e-5) * scale
    assert rel_err(got[B.FORM_AUTO], want) < (1e-12 if prec == "f64" else 2e-5)
    assert gs.sync() == (0, 0)
    gs.close()


def test_device_driven_run_with_data_in_a_graph():
    """advance() takes the data's times from the device: graph replays equal
    eager steps bit for bit and reach the oracle's state."""
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    bcs = dict(zip("WESN", (PROD, OUT, SINE, OUT)))
    gs, dg = make_pair_2d(40, 24, (-1, 1, -1, 1), 2, "Q", "advection", "ssprk3", bcs, "f64", beta=(1.0, 1.0))
    u = inp.random_modal_state(24, 40, 2, "Q", "advection", seed=8)
    stream = torch.cuda.Stream()
    out = []
    for capture in (False, True):
        s = B.Solver(gs.mesh, 2, B.BASIS_Q, T.SSPRK3, B.ADVECTION, B.F64, beta=(1.0, 1.0), stream=stream.cuda_stream)
        s.set_state(to_planes(u), 0.0)
        for _ in range(2):
            s.advance(3, 0.05, 10.0, capture=capture)
        out.append((s.get_state(), s.time()))
        s.close()
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
    dt = 0.05 / (1.0 / dg.dx + 1.0 / dg.dy)
    want, t = u, 0.0
    for _ in range(6):
        want = step2d(dg, want, t, dt, TAB_NAMES["ssprk3"])
        t += dt
    assert rel_err(from_planes(out[0][0]), want) < 1e-12
    gs.close()


@pytest.mark.parametrize("nx", [1, 2, 29, 30, 31, 61, 240, 241, 930, 960])
@pytest.mark.parametrize("physics,beta,bcs", [("advection", 1.0, (PER, PER)), ("advection", -0.7, (PER, PER)),
                                              ("advection", 1.0, (("sine", 1.0, 1.0, 0.0, 1.0, 0.0), OUT)),
                                              ("advection", -1.0, (OUT, CONST)), ("euler", 1.0, (PER, PER)),
                                              ("euler", 1.0, (OUT, ("const", [1.0, 0.4, 2.6])))])
def test_1d_runs(nx, physics, beta, bcs):
    k, n, tab = (2, 7, "ssprk3") if nx % 2 else (3, 6, "rk4")
    gs, dg = make_pair_1d(nx, (0, 2 * np.pi), k, physics, tab, bcs, "f64", beta=beta)
    u = inp.random_modal_state_1d(nx, k, 3 if physics == "euler" else 1, seed=nx)
    dt = 0.02 * 2 * np.pi / nx
    gs.set_state(to_planes(u), 0.0)
    gs.run_fixed(n, dt)
    a = gs.get_state()
    gs.set_state(to_planes(u), 0.0)
    for _ in range(n):
        gs.step(dt)
    assert np.array_equal(a, gs.get_state())
    w, t = u.copy(), 0.0
    for _ in range(n):
        w = step1d(dg, w, t, dt, TAB_NAMES[tab])
        t += dt
    assert rel_err(from_planes(a, 1), w) < 1e-12
    gs.close()
