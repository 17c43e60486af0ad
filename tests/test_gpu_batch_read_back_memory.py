"""Reading an FP32 problem of a batch back where the device has no room for its
FP64 values: they are widened on the host, to the same numbers."""
import numpy as np
import pytest

import crkdg_inputs as inp
from tests.pairing import to_planes

pytestmark = pytest.mark.gpu
NX, NY = 900, 640
VALUES = NX * NY * 24     # 55 MB in FP32, 111 MB in FP64


@pytest.mark.parametrize("limited", [False, True])
def test_read_back_with_little_memory(limited):
    import torch
    from paper_2307_06471_gb300 import binding as B
    from paper_2307_06471_gb300 import tableaux as T
    stream = torch.cuda.Stream()
    u = to_planes(inp.random_modal_state(NY, NX, 2, "P", "euler", seed=3, amp=0.2))

    def batch():
        b = B.Batch([(NX, NY, (0.0, 1.0, 0.0, 1.0))], 2, B.BASIS_P, T.SSPRK3, B.F32, stream=stream.cuda_stream)
        b.set_state(0, u)
        if limited:
            b.limit(1.0)
        return b
    a, b = batch(), batch()
    want = a.get_state(0)
    a.close()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - VALUES * 6, dtype=torch.uint8, device="cuda")
    try:
        assert np.array_equal(b.get_state(0), want)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert np.array_equal(b.get_state(0), want)
    b.close()
