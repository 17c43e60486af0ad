"""The modal steps of linear advection with weights b that do not sum to one (the
tableau is the caller's): every side's exterior trace counts sum_i b_i of its
stages' values, as in the quadrature form.  Bands: the parity tests'."""
import numpy as np
import pytest

import crkdg_inputs as inp
from oracle import tableaux as OTB
from oracle.dg1d import crkdg_step as step1d
from oracle.dg2d import crkdg_step as step2d
from tests.pairing import from_planes, make_pair_1d, make_pair_2d, rel_err, to_planes

pytestmark = pytest.mark.gpu
A, W = [[0.0, 0.0, 0.0], [0.5, 0.0, 0.0], [0.25, 0.5, 0.0]], [0.3, 0.4, 0.2]
SINE, OUT, CONST = ("sine", 0.8, 2.0, 1.5, 3.0, 0.3), ("outflow",), ("const", [0.4])


@pytest.fixture()
def tab(monkeypatch):
    from paper_2307_06471_gb300 import tableaux as GTB
    monkeypatch.setitem(GTB.BY_NAME, "short", (A, W))
    return OTB.tableau(A, W)


@pytest.mark.parametrize("beta", [1.0, -1.0])
@pytest.mark.parametrize("bcs", [(OUT, OUT), (CONST, CONST), (("sine", 1.0, 1.0, 0.0, 1.0, 0.0), OUT)])
def test_1d(tab, bcs, beta):
    nx, n = 50, 5
    gs, dg = make_pair_1d(nx, (0, 1), 2, "advection", "short", bcs, "f64", beta=beta)
    u = inp.random_modal_state_1d(nx, 2, 1, seed=3)
    dt = 0.02 / nx
    gs.set_state(to_planes(u), 0.0)
    gs.run_fixed(n, dt)
    w, t = u.copy(), 0.0
    for _ in range(n):
        w = step1d(dg, w, t, dt, tab)
        t += dt
    assert rel_err(from_planes(gs.get_state(), 1), w) < 1e-12
    gs.close()


@pytest.mark.parametrize("beta", [(1.0, 0.5), (-1.0, -0.5)])
@pytest.mark.parametrize("sides", [(CONST, CONST, CONST, CONST), (SINE, CONST, OUT, SINE), (OUT, OUT, OUT, OUT)])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_2d(tab, sides, beta, prec):
    from paper_2307_06471_gb300 import binding as B
    nx, ny = 37, 21
    gs, dg = make_pair_2d(nx, ny, (-1, 1, -0.6, 1), 2, "Q", "advection", "short", dict(zip("WESN", sides)), prec, beta=beta)
    u = inp.random_modal_state(ny, nx, 2, "Q", "advection", seed=nx)
    dt = 0.01 / nx
    want, t = u, 0.25
    for _ in range(3):
        want = step2d(dg, want, t, dt, tab)
        t += dt
    for form in (B.FORM_AUTO, B.FORM_QUADRATURE):
        gs.set_operator_form(form)
        gs.set_state(to_planes(u), 0.25)
        for _ in range(3):
            gs.step(dt)
        assert rel_err(from_planes(gs.get_state()), want) < (1e-12 if prec == "f64" else 2e-5)
    gs.close()
