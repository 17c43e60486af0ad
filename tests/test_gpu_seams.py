"""The quadrature step with seams (the faces between a strip's segments formed
by launches of their own) against the oracle and against the step that
recomputes halo rows: segments of one row, of one and two rows mixed, of a few
and of the whole mesh, periodic and wall / constant-state / moving-shock sides,
ragged columns, the limit on load, batches.  The segments do not change a
result, bit for bit; the oracle bands are the parity tests' (FP64 1e-13 a step
and 1e-12 for three, the deviation form 3e-7 of the state)."""
import numpy as np
import pytest

import crkdg_inputs as inp
from oracle.dg2d import cfl_dt_2d, crkdg_step
from oracle.limiter import tvb_limit
from tests.pairing import TAB_NAMES, from_planes, make_pair_2d, rel_err, to_planes

pytestmark = pytest.mark.gpu
PER = {s: ("periodic",) for s in "WESN"}
STATE = [1.0, 0.3, -0.2, 2.4]
WALLS = {"W": ("const", STATE), "E": ("outflow",), "S": ("reflect",), "N": ("reflect",)}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2307_06471_gb300 import build
    build.build()


@pytest.mark.parametrize("bcs", [PER, WALLS], ids=["periodic", "walls"])
@pytest.mark.parametrize("ny", [1, 2, 3, 11, 20])
@pytest.mark.parametrize("prec,k,basis,tab", [("f64", 2, "P", "ssprk3"), ("f64", 2, "Q", "rk4"), ("f64", 1, "Q", "midpoint"),
                                              ("f32d", 2, "Q", "rk4"), ("f32", 2, "Q", "rk4"), ("f32", 3, "P", "rk4")])
def test_segments_do_not_change_the_step(prec, k, basis, tab, ny, bcs):
    nx = 37
    gs, dg = make_pair_2d(nx, ny, (0, 1, 0, 1.1 * ny / nx), k, basis, "euler", tab, bcs, prec)
    u = inp.random_modal_state(ny, nx, k, basis, "euler", seed=ny)
    if prec != "f64":
        u = from_planes(to_planes(u).astype(np.float32).astype(np.float64))
    dt = 0.2 * cfl_dt_2d(dg, u, 1.0)
    want, t = u, 0.0
    for _ in range(3):
        want = crkdg_step(dg, want, t, dt, TAB_NAMES[tab])
        t += dt
    first = None
    for rows in sorted({1, 2, 3, 4, 6, 7, ny}):
        gs.set_launch(min(rows, ny), 1 + rows % 2)
        gs.set_state(to_planes(u), 0.0)
        for _ in range(3):
            gs.step(dt)
        got = gs.get_state()
        first = got if first is None else first
        assert np.array_equal(got, first), rows
    assert rel_err(from_planes(first), want) < {"f64": 1e-12, "f32d": 1e-6, "f32": 2e-5}[prec]
    assert gs.sync() == (0, 0)
    assert gs.step_count() == 3 * len({1, 2, 3, 4, 6, 7, ny})
    gs.close()


@pytest.mark.parametrize("rows", [1, 3, 29])
def test_limit_on_load_with_seams_f64(rows):
    from paper_2307_06471_gb300 import binding as B
    nx, ny = 41, 29
    gs, dg = make_pair_2d(nx, ny, (0, 1, 0, 1), 2, "P", "euler", "ssprk3", PER, "f64")
    u = inp.random_modal_state(ny, nx, 2, "P", "euler", seed=4, amp=0.2)
    gs.set_limit_mode(B.LIMIT_FUSED)
    gs.set_launch(rows, 1)
    gs.set_state(to_planes(u), 0.0)
    gs.limit(500.0)
    dt = 0.2 * cfl_dt_2d(dg, u, 1.0)
    lim = lambda v, t: tvb_limit(dg, v, 500.0, t)[0]
    want = crkdg_step(dg, lim(u, 0.0), 0.0, dt, TAB_NAMES["ssprk3"], limiter=lim)
    gs.step(dt)
    assert rel_err(from_planes(gs.get_state()), want) < 1e-12
    gs.close()


@pytest.mark.parametrize("prec,basis,tab", [("f64", "P", "ssprk3"), ("f32", "Q", "rk4")])
def test_batch_segments(prec, basis, tab):
    """Problems of uneven sizes, one of a single row; one reaches t_end first
    and then costs nothing."""
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    sizes = [(37, 1), (31, 12), (64, 33)]
    stream = torch.cuda.Stream()
    outs = []
    for rows in (1, 3, 40):
        b = B.Batch([(nx, ny, (0.0, 1.0, 0.0, ny / nx)) for nx, ny in sizes], 2, B.BASIS_P if basis == "P" else B.BASIS_Q,
                    T.BY_NAME[tab], B.F64 if prec == "f64" else B.F32, bc=(B.BC_PERIODIC,) * 4, stream=stream.cuda_stream)
        b.set_launch(rows, 2)
        for i, (nx, ny) in enumerate(sizes):
            b.set_state(i, to_planes(inp.random_modal_state(ny, nx, 2, basis, "euler", seed=i)))
        done = b.run(0.1, 0.02, steps_per_graph=6, max_graphs=3)
        info = [b.info(i) for i in range(3)]
        outs.append([b.get_state(i) for i in range(3)] + [[x[0] for x in info], [x[1] for x in info], done])
        assert all(x[2] == 0 for x in info)
        b.close()
    for o in outs[1:]:
        for x, y in zip(o, outs[0]):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("case", ["mode", "linear"])
def test_first_step_can_be_captured(case):
    """A step allocates nothing: the first one on a context, and the first
    after a change of the limit mode, are captured on the caller's stream; a
    graph captured in the other mode stays valid.  Bitwise equal to steps that
    are not captured."""
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    phys = "euler" if case == "mode" else "advection"
    nx, ny = 333, 200
    mesh = B.make_mesh(2, nx, ny, (0.0, 1.0, 0.0, 0.6), [B.BC_PERIODIC] * 4)
    u = to_planes(inp.random_modal_state(ny, nx, 2, "P", phys, seed=9))
    dt = 0.02 / nx
    torch.zeros(1, device="cuda")
    stream = torch.cuda.Stream()

    def solver():
        s = B.Solver(mesh, 2, B.BASIS_P, T.SSPRK3, B.EULER if case == "mode" else B.ADVECTION, B.F64, stream=stream.cuda_stream)
        s.set_state(u, 0.0)
        return s
    plain, captured = solver(), solver()
    graphs = []
    for mode in ((B.LIMIT_PASS, B.LIMIT_FUSED) if case == "mode" else (B.LIMIT_PASS, B.LIMIT_PASS)):
        for s in (plain, captured):
            if case == "mode":
                s.set_limit_mode(mode)
                s.limit(50.0)
        plain.step(dt)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            captured.step(dt)
        graphs.append(g)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for g in graphs:
            g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(captured.get_state(), plain.get_state())
    captured.close()
    plain.close()
