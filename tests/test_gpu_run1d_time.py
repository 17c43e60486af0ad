"""A 1D run's clock goes on as its stage times did: runs in parts, one run and
single steps end at the same time and, with boundary data that depend on it, in
the same state."""
import numpy as np
import pytest

import crkdg_inputs as inp
from tests.pairing import make_pair_1d, to_planes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [40, 1000])       # a run in one launch; one launch a step
def test_runs_in_parts(nx):
    gs, _ = make_pair_1d(nx, (0, 1), 2, "advection", "ssprk3", (("sine", 1.0, 1.0, 0.0, 9.0, 0.0), ("outflow",)), "f64")
    u = to_planes(inp.random_modal_state_1d(nx, 2, 1, seed=5))
    dt = 0.1 / 3 / nx
    out = []
    for parts in ([97], [31, 66], [1, 95, 1], [1] * 97):
        gs.set_state(u, 0.1)
        for n in parts:
            if parts == [1] * 97:
                gs.step(dt)
            else:
                gs.run_fixed(n, dt)
        out.append((gs.time(), gs.get_state()))
    for t, s in out[1:]:
        assert t == out[0][0] and np.array_equal(s, out[0][1])
    gs.close()
