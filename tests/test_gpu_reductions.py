"""The FP64 reductions of the cell averages (crkdg_cfl_dt, crkdg_conservation,
the first dt of a batch): cells that cannot hold the maximum wave speed are
sorted out by an FP32 estimate, so the cases are those where the estimate
could mislead -- near ties, uniform states, a pressure that is a small
difference of large energies, values an FP32 number cannot hold -- at sizes
around the 1024-cell chunks of a block, against the formula in numpy FP64.

Tolerance: the kernel evaluates the same formula in FP64; about 12 roundings
of 1.1e-16, amplified in the pressure by E / p (1e3 in the cold state, half
of it in the sound speed): 1e-13 relative.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (33, 31), (32, 32), (41, 25), (700, 613)]
STATES = ["random", "uniform", "near_tie", "cold", "huge"]


def averages(kind, nx, ny, seed):
    rng = np.random.default_rng(seed)
    n = (ny, nx)
    rho, p = 1 + 0.3 * rng.uniform(-1, 1, n), 1 + 0.3 * rng.uniform(-1, 1, n)
    w, v = rng.uniform(-1, 1, n), rng.uniform(-1, 1, n)
    if kind == "uniform":
        rho, p, w, v = (np.full(n, a.flat[0]) for a in (rho, p, w, v))
    elif kind == "near_tie":
        rho, p, w, v = (np.full(n, a.flat[0]) * (1 + 1e-6 * rng.uniform(-1, 1, n)) for a in (rho, p, w, v))
    elif kind == "cold":
        p = 1e-3 * p
    s = 1e30 if kind == "huge" else 1.0
    E = p / 0.4 + 0.5 * rho * (w * w + v * v)
    return np.stack([rho, rho * w, rho * v, E]) * s


def speed(a, dx, dy):
    w, v = a[1] / a[0], a[2] / a[0]
    p = 0.4 * (a[3] - 0.5 * (a[1] * w + a[2] * v))
    c = np.sqrt(np.maximum(1.4 * p / a[0], 0.0))
    return np.max((np.abs(w) + c) / dx + (np.abs(v) + c) / dy)


@pytest.mark.parametrize("precision", ["f32", "f64", "f32d"])
@pytest.mark.parametrize("kind", STATES)
@pytest.mark.parametrize("size", SIZES)
def test_speed_and_totals_2d(size, kind, precision):
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    nx, ny = size
    dx, dy = 0.01, 0.013
    a = averages(kind, nx, ny, 5)
    if precision == "f32":
        a = a.astype(np.float32).astype(np.float64)
    mesh = B.make_mesh(2, nx, ny, (0.0, nx * dx, 0.0, ny * dy), [B.BC_OUTFLOW] * 4)
    s = B.Solver(mesh, 1, B.BASIS_P, T.HEUN2, B.EULER, {"f32": B.F32, "f64": B.F64, "f32d": B.F32D}[precision])
    u = np.zeros(s.shape)
    u[:, 0] = a
    s.set_state(u)
    if precision == "f32d":
        a = s.get_state()[:, 0]      # hi + lo
    dx, dy = nx * dx / nx, ny * dy / ny
    want = speed(a, dx, dy)
    assert abs(0.25 / s.cfl_dt(0.25) - want) <= 1e-13 * want
    tot = [math.fsum(a[v].ravel()) * dx * dy for v in range(4)]
    mag = [math.fsum(np.abs(a[v]).ravel()) * dx * dy for v in range(4)]
    got = s.conservation()
    assert all(abs(got[v] - tot[v]) <= 1e-13 * mag[v] for v in range(4))
    assert s.sync() == (0, 0)
    s.close()


@pytest.mark.parametrize("bad", ["nan", "vacuum", "negative"])
def test_status_of_a_bad_cell(bad):
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    nx, ny = 77, 31
    a = averages("random", nx, ny, 9)
    good = a.copy()
    y, x = 30, 76
    if bad == "nan":
        a[3, y, x] = np.nan
    elif bad == "vacuum":
        a[:, y, x] = 0.0
    else:
        a[3, y, x] = 0.0
        a[1, y, x] = a[2, y, x] = 1e-3     # p < 0, c = 0: slower than the rest
    mesh = B.make_mesh(2, nx, ny, (0.0, 1.0, 0.0, 1.0), [B.BC_OUTFLOW] * 4)
    s = B.Solver(mesh, 1, B.BASIS_P, T.HEUN2, B.EULER, B.F32)
    u = np.zeros(s.shape)
    u[:, 0] = a
    s.set_state(u)
    good = good.astype(np.float32).astype(np.float64)
    keep = np.ones((ny, nx), bool)
    keep[y, x] = False
    want = speed(good[:, keep], 1.0 / nx, 1.0 / ny)
    assert abs(0.25 / s.cfl_dt(0.25) - want) <= 1e-13 * want      # the bad cell does not show in the maximum
    code, st = s.sync()
    assert code == B.ENONPHYSICAL and st & (B.ST_NONPHYSICAL | B.ST_NAN)
    s.close()


@pytest.mark.parametrize("nx", [1, 1023, 1024, 1025, 9000])
def test_speed_1d(nx):
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    rng = np.random.default_rng(nx)
    rho, p, w = 1 + 0.3 * rng.uniform(-1, 1, nx), 1 + 0.3 * rng.uniform(-1, 1, nx), rng.uniform(-1, 1, nx)
    mesh = B.make_mesh(1, nx, 1, (0.0, 1.0, 0.0, 1.0), [B.BC_PERIODIC] * 4)
    s = B.Solver(mesh, 1, B.BASIS_P, T.HEUN2, B.EULER, B.F64)
    u = np.zeros(s.shape)
    u[0, 0, 0], u[1, 0, 0], u[2, 0, 0] = rho, rho * w, p / 0.4 + 0.5 * rho * w * w
    s.set_state(u)
    want = np.max(np.abs(w) + np.sqrt(1.4 * p / rho)) * nx
    assert abs(0.25 / (s.cfl_dt(0.25)) - want) <= 1e-13 * want
    s.close()


def test_batch_first_dt():
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    sizes = [(1, 1), (33, 31), (150, 140)]
    stream = torch.cuda.Stream()
    b = B.Batch([(nx, ny, (0.0, 1.0, 0.0, 1.0)) for nx, ny in sizes], 1, B.BASIS_P, T.HEUN2, B.F32, stream=stream.cuda_stream)
    want = []
    for i, (nx, ny) in enumerate(sizes):
        a = averages("random", nx, ny, i).astype(np.float32).astype(np.float64)
        u = np.zeros((4, 3, ny, nx))
        u[:, 0] = a
        b.set_state(i, u)
        want.append(0.05 / speed(a, 1.0 / nx, 1.0 / ny))
    b.run(0.05, 1.0, steps_per_graph=1)
    for i, dt in enumerate(want):
        t, n, _ = b.info(i)
        assert n == 1 and abs(t - dt) <= 1e-13 * dt
    b.close()
