"""The batch's autotuner starts from the shape the batch has and knows the short
segments that its default takes on small ensembles: tuning does not make a step
slower, and leaves the states as they are.  (On this ensemble a step of 8-row
segments takes several times one of the default's.)"""
import numpy as np
import pytest

import crkdg_inputs as inp
from tests.pairing import to_planes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_tuning_a_small_ensemble(prec):
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    stream = torch.cuda.Stream()
    sizes = [(48, 48), (40, 50), (60, 33)]
    b = B.Batch([(nx, ny, (0.0, 1.0, 0.0, ny / nx)) for nx, ny in sizes], 2, B.BASIS_Q, T.RK4,
                B.F64 if prec == "f64" else B.F32, bc=(B.BC_PERIODIC,) * 4, stream=stream.cuda_stream)
    for i, (nx, ny) in enumerate(sizes):
        b.set_state(i, to_planes(inp.random_modal_state(ny, nx, 2, "Q", "euler", seed=i)))

    def step_ms():
        b.run(0.02, 1e6, steps_per_graph=20)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        times = []
        with torch.cuda.stream(stream):
            for _ in range(5):
                e0.record(stream)
                b.run(0.02, 1e6, steps_per_graph=20)
                e1.record(stream)
                stream.synchronize()
                times.append(e0.elapsed_time(e1))
        return sorted(times)[2]
    before = step_ms()
    states = [b.get_state(i) for i in range(3)]
    assert b.autotune(0.02) > 0.0
    assert all(np.array_equal(b.get_state(i), states[i]) for i in range(3))
    assert step_ms() <= 1.25 * before
    b.close()
