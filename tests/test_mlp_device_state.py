"""The network's kernels take more shared memory than a launch may ask for
without their attribute, which belongs to a device: a call that may be the first
on its device sets it (as the tcgen05 inference does), and nothing of the network
is decided once for the process."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_attributes_are_set_by_every_call():
    src = open(os.path.join(ROOT, "paper_2307_06471_gb300", "csrc", "mlp.cu")).read()
    src = re.sub(r"//[^\n]*", "", src)
    assert "call_once" not in src and "once_flag" not in src
    for entry in ("int crkdg_mlp_predict(", "int crkdg_mlp_predict_tc(", "static int train_workspace("):
        body = src[src.index(entry):]
        assert "cudaFuncSetAttribute(" in body[:body.index("\n}\n")], entry
