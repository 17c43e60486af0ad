"""The step's shared row helpers index the basis tables by constants only: a copy
of the Q^3 table (12.7 KB) on every thread's stack is what an index that is not
folded costs, in the step and in the seam kernels.  Compiled alone, with the
registers of a whole row."""
import re
import shutil
import subprocess

import pytest

from paper_2307_06471_gb300 import build

SRC = """
#include "step2d.cuh"
namespace crk {
template <class T, int K, int B, bool COMP, bool DEV>
__global__ void __launch_bounds__(256) row(const T* __restrict__ in, T* __restrict__ out) {
    constexpr int NM = Tab2D<K, B>::NM, NQ = K + 1;
    T P[NM], V[NM], un[NM], FS[NQ], FN[NQ];
    for (int m = 0; m < NM; ++m) {
        P[m] = in[m * 256 + threadIdx.x];
        V[m] = in[(NM + m) * 256 + threadIdx.x];
        un[m] = in[(2 * NM + m) * 256 + threadIdx.x];
    }
    for (int p = 0; p < NQ; ++p) {
        FS[p] = in[(3 * NM + p) * 256 + threadIdx.x];
        FN[p] = in[(3 * NM + NQ + p) * 256 + threadIdx.x];
    }
    row_update<T, K, B, COMP, false>(P, P, V, FS, un, T(2), T(3), T(4));
    add_north<T, K, B, DEV>(P, FN, T(5), T(3), T(4));
    for (int m = 0; m < NM; ++m) out[m * 256 + threadIdx.x] = P[m];
}
template __global__ void row<float, 3, 1, false, false>(const float*, float*);
template __global__ void row<float, 3, 1, true, true>(const float*, float*);
template __global__ void row<double, 3, 1, false, false>(const double*, double*);
template __global__ void row<double, 2, 1, false, false>(const double*, double*);
}  // namespace crk
"""


@pytest.mark.skipif(shutil.which(build.NVCC) is None, reason="needs nvcc")
def test_row_helpers_leave_no_table_on_the_stack(tmp_path):
    src = tmp_path / "row.cu"
    src.write_text(SRC)
    cmd = [build.NVCC] + build.ARCH + build.FLAGS + ["-I", build.CSRC, "-Xptxas", "-v", "-c", str(src), "-o", str(tmp_path / "row.o")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    stacks = [int(x) for x in re.findall(r"(\d+) bytes stack frame", r.stderr)]
    assert len(stacks) == 4 and max(stacks) == 0, stacks
