"""Where the 2D step leaves the faces between segments to launches of their own:
the rule of common.cuh on shapes that were measured both ways (a host program
around the rule; 152 SMs), forward-Euler passes of the original RKDG among them."""
import os
import shutil
import subprocess

import pytest

from paper_2307_06471_gb300 import build

SMS = 152
# (what, element size, stages, modes, face points, variables, deviation form, limit on load, ny, segments, strips, seams)
CASES = [
    ("P2 SSP-RK3 96^2, a row each", 4, 3, 6, 3, 4, 0, 0, 96, 96, 4, False),
    ("P2 SSP-RK3 400^2, 5 rows", 4, 3, 6, 3, 4, 0, 0, 400, 80, 14, False),
    ("P2 SSP-RK3 1920x480, a row each, many waves", 4, 3, 6, 3, 4, 0, 0, 480, 480, 64, True),
    ("P2 SSP-RK3 1920x480, 26 rows", 4, 3, 6, 3, 4, 0, 0, 480, 19, 64, False),
    ("P1 SSP-RK3 96^2", 4, 3, 3, 2, 4, 0, 0, 96, 96, 4, False),
    ("Q2 SSP-RK3 96^2, a row each, few warps", 4, 3, 9, 3, 4, 0, 0, 96, 96, 4, False),
    ("Q2 SSP-RK3 128^2, a row each", 4, 3, 9, 3, 4, 0, 0, 125, 125, 5, True),
    ("Q2 SSP-RK3 400^2, 5 rows", 4, 3, 9, 3, 4, 0, 0, 400, 80, 14, False),
    ("Q2 RK4 96^2", 4, 4, 9, 3, 4, 0, 0, 96, 96, 4, True),
    ("Q2 RK4 400^2, 5 rows", 4, 4, 9, 3, 4, 0, 0, 400, 80, 14, True),
    ("Q2 RK4 640^2, 12 rows", 4, 4, 9, 3, 4, 0, 0, 640, 54, 22, False),
    ("P3 RK4 1280^2, 46 rows", 4, 4, 10, 4, 4, 0, 0, 1280, 28, 43, True),
    ("Q3 RK4 400^2", 4, 4, 16, 4, 4, 0, 0, 400, 80, 14, True),
    ("deviation Q2 RK4 320^2, 3 rows", 4, 4, 9, 3, 4, 1, 0, 320, 107, 11, True),
    ("deviation Q2 RK4 400^2, 5 rows", 4, 4, 9, 3, 4, 1, 0, 400, 80, 14, False),
    ("deviation Q2 RK4 1280^2, 46 rows", 4, 4, 9, 3, 4, 1, 0, 1280, 28, 43, False),
    ("advection Q2 SSP-RK3 96^2", 4, 3, 9, 3, 1, 0, 0, 96, 96, 4, False),
    ("advection Q2 RK4 256^2, a row each", 4, 4, 9, 3, 1, 0, 0, 253, 253, 9, True),
    ("advection Q2 RK4 400^2, 3 rows", 4, 4, 9, 3, 1, 0, 0, 400, 134, 14, False),
    ("forward Euler Q2 96^2", 4, 1, 9, 3, 4, 0, 0, 96, 96, 4, False),
    ("forward Euler P2 400^2", 4, 1, 6, 3, 4, 0, 0, 400, 80, 14, False),
    ("forward Euler Q3 96^2", 4, 1, 16, 4, 4, 0, 0, 96, 96, 4, True),
    ("limit on load, FP32", 4, 4, 9, 3, 4, 0, 1, 96, 96, 4, False),
    ("FP64 whatever the shape", 8, 1, 3, 2, 4, 0, 0, 640, 1, 22, True),
    ("FP64, limit on load", 8, 3, 6, 3, 4, 0, 1, 640, 160, 22, True),
]


@pytest.mark.skipif(shutil.which(build.NVCC) is None, reason="needs nvcc")
def test_measured_shapes(tmp_path):
    lines = ["    std::puts(crk::use_seams(%d, %d, %d, %d, %d, %d, %d, %d, %d, %dLL, %d) ? \"1\" : \"0\");" %
             (es, s, nm, nq, nv, dev, lim, ny, segs, strips * segs, SMS)
             for _, es, s, nm, nq, nv, dev, lim, ny, segs, strips, _ in CASES]
    src = tmp_path / "rule.cu"
    src.write_text('#include <cstdio>\n#include "common.cuh"\nint main() {\n' + "\n".join(lines) + "\n    return 0;\n}\n")
    exe = tmp_path / "rule"
    r = subprocess.run([build.NVCC] + build.ARCH + build.FLAGS + ["-I", build.CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert [(c[0], o == "1") for c, o in zip(CASES, out)] == [(c[0], c[-1]) for c in CASES]
