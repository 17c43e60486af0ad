"""The maximum wave speed for ratios of specific heats far from 1.4: the FP32
estimate that sorts cells out loses accuracy with (gamma - 1) where the energy is
mostly kinetic, and must leave such cells to the FP64 formula.  Cells of nearly
equal speed, each nearly all kinetic energy.

Tolerance: about 12 roundings of 1.1e-16 in the FP64 formula, amplified in p by E
/ (E - KE) <= 1 / (0.9 THIN), half of it in the sound speed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
THIN = 1.5e-4             # internal energy as a part of E
TOL = 0.5 * 12 * 1.1e-16 / (0.9 * THIN)


def averages(n, seed):
    """Cells whose speeds differ by parts in a thousand."""
    rng = np.random.default_rng(seed)
    rho = 1 + 0.3 * rng.uniform(-1, 1, n)
    w, v = 1 + 1e-3 * rng.uniform(-1, 1, n), 1 + 1e-3 * rng.uniform(-1, 1, n)
    ke = 0.5 * rho * (w * w + v * v)
    return np.stack([rho, rho * w, rho * v, ke / (1 - THIN * (1 + 1e-2 * rng.uniform(-1, 1, n)))])


def speed(a, gamma, dx, dy):
    w, v = a[1] / a[0], a[2] / a[0]
    p = (gamma - 1) * (a[3] - 0.5 * (a[1] * w + a[2] * v))
    c = np.sqrt(np.maximum(gamma * p / a[0], 0.0))
    return np.max((np.abs(w) + c) / dx + (np.abs(v) + c) / dy)


@pytest.mark.parametrize("gamma", [1.005, 1.4, 5.0 / 3.0, 3.0, 8.0, 100.0, 1000.0])
@pytest.mark.parametrize("seed", range(4))
def test_maximum_speed(gamma, seed):
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    nx, ny = 97, 83
    dx, dy = 0.01, 0.013
    a = averages((ny, nx), seed)
    mesh = B.make_mesh(2, nx, ny, (0.0, nx * dx, 0.0, ny * dy), [B.BC_OUTFLOW] * 4)
    s = B.Solver(mesh, 1, B.BASIS_P, T.HEUN2, B.EULER, B.F64, gamma=gamma)
    u = np.zeros(s.shape)
    u[:, 0] = a
    s.set_state(u)
    want = speed(a, gamma, nx * dx / nx, ny * dy / ny)
    assert abs(0.25 / s.cfl_dt(0.25) - want) <= TOL * want
    s.close()
    stream = torch.cuda.Stream()
    b = B.Batch([(nx, ny, (0.0, nx * dx, 0.0, ny * dy))], 1, B.BASIS_P, T.HEUN2, B.F64, gamma=gamma, stream=stream.cuda_stream)
    b.set_state(0, u)
    b.run(1e-9, 1.0, steps_per_graph=1)
    t, n, _ = b.info(0)
    assert n == 1 and abs(1e-9 / t - want) <= TOL * want
    b.close()
