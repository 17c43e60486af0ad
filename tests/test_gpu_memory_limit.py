"""Contexts on a device with little memory left: the seam scratch of the 2D step
(up to 256 MiB or an eighth of a state copy) gives way -- fewer segments in FP64,
recomputed halo rows in FP32 -- and the steps stay the same bit for bit."""
import numpy as np
import pytest

import crkdg_inputs as inp
from tests.pairing import to_planes

pytestmark = pytest.mark.gpu
ROOM = 160 << 20          # left free: less than the scratch asks for, more than half of it


def _run(s, u, dt):
    s.set_launch(1, 0)
    s.set_state(u, 0.0)
    for _ in range(2):
        s.step(dt)
    return s.get_state()


@pytest.mark.parametrize("prec,basis,tab", [("f64", "P", "ssprk3"), ("f32d", "Q", "rk4")])
def test_seam_scratch_gives_way(prec, basis, tab):
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    nx, ny = 1024, 400
    mesh = B.make_mesh(2, nx, ny, (0.0, 2.56, 0.0, 1.0), [B.BC_PERIODIC] * 4)
    args = (mesh, 2, B.BASIS_P if basis == "P" else B.BASIS_Q, T.BY_NAME[tab], B.EULER, B.F64 if prec == "f64" else B.F32D)
    u = to_planes(inp.random_modal_state(ny, nx, 2, basis, "euler", seed=7))
    n = B.state_bytes(mesh, args[1], args[2], args[4], args[5])
    free0 = torch.cuda.mem_get_info()[0]
    bufs = [torch.zeros(n, dtype=torch.uint8, device="cuda") for _ in range(2)]
    ptrs = tuple(b.data_ptr() for b in bufs)
    a = B.Solver(*args, state_buffers=ptrs)
    want = _run(a, u, 1e-5)
    taken = free0 - torch.cuda.mem_get_info()[0]
    assert taken >= 3 * ROOM // 2            # the scratch does ask for more than ROOM (with the states)
    b = B.Solver(*args, state_buffers=ptrs)
    b.set_state(u, 0.0)                      # (its staging buffer, where it has one)
    a.close()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - ROOM, dtype=torch.uint8, device="cuda")
    try:
        got = _run(b, u, 1e-5)
        c = B.Solver(*args, state_buffers=ptrs)      # creation, too
        c.close()
    finally:
        del hog
        torch.cuda.empty_cache()
    assert np.array_equal(got, want) and b.sync() == (0, 0)
    assert np.array_equal(_run(b, u, 1e-5), want)    # with the whole room again
    b.close()


def test_autotune_keeps_the_scratch_of_its_choice_only():
    """Trials of short segments ask for scratch that the kept shape does not
    need: what the context gives back at its end is what one that was set to the
    kept shape gives back."""
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    nx, ny = 240, 4000
    mesh = B.make_mesh(2, nx, ny, (0.0, 0.6, 0.0, 10.0), [B.BC_PERIODIC] * 4)
    u = to_planes(inp.random_modal_state(ny, nx, 2, "P", "euler", seed=7))

    def held(s):
        s.set_state(u, 0.0)
        s.step(1e-5)
        s.sync()
        free = torch.cuda.mem_get_info()[0]
        s.close()
        return torch.cuda.mem_get_info()[0] - free

    def solver():
        return B.Solver(mesh, 2, B.BASIS_P, T.SSPRK3, B.EULER, B.F64)
    tuned, plain = solver(), solver()
    tuned.set_state(u, 0.0)
    tuned.autotune()
    plain.set_launch(*tuned.get_launch())
    assert held(tuned) <= held(plain) + (8 << 20)
