"""A batch on a device with little memory left: its seam scratch gives way (halo
rows in FP32, fewer segments in FP64), the steps stay the same bit for bit, and
a change of launch shape or limit mode always leaves tables that can be run."""
import numpy as np
import pytest

import crkdg_inputs as inp
from tests.pairing import to_planes

pytestmark = pytest.mark.gpu
ROOM = 160 << 20          # left free: less than the seam scratch asks for (256 MiB)
SIZES = [(512, 400), (300, 500), (640, 160), (37, 1)]


@pytest.mark.parametrize("prec,basis,tab", [("f64", "P", "ssprk3"), ("f32", "Q", "rk4")])
def test_batch_scratch_gives_way(prec, basis, tab):
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    stream = torch.cuda.Stream()
    states = [to_planes(inp.random_modal_state(ny, nx, 2, basis, "euler", seed=i)) for i, (nx, ny) in enumerate(SIZES)]

    def run(b, rows):
        b.set_launch(rows, 2)
        for i, u in enumerate(states):
            b.set_state(i, u)
        b.run(0.1, 1e6, steps_per_graph=3)
        return [b.get_state(i) for i in range(len(SIZES))]
    b = B.Batch([(nx, ny, (0.0, 1.0, 0.0, ny / nx)) for nx, ny in SIZES], 2, B.BASIS_P if basis == "P" else B.BASIS_Q,
                T.BY_NAME[tab], B.F64 if prec == "f64" else B.F32, bc=(B.BC_PERIODIC,) * 4, stream=stream.cuda_stream)
    want = run(b, 1)
    b.set_launch(40, 2)
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - ROOM, dtype=torch.uint8, device="cuda")
    try:
        got = [run(b, 1), run(b, 3)]
        b.set_limit_mode(B.LIMIT_FUSED)      # (nothing pending: the same steps)
        got.append(run(b, 1))
    finally:
        del hog
        torch.cuda.empty_cache()
    for g in got:
        for x, y in zip(g, want):
            assert np.array_equal(x, y)
    b.close()
