// The modal step for linear advection (step2d_linear.cuh), FP32 and FP64,
// for every (k, basis), and its launcher.
#include "launch.h"
#include "step2d_linear.cuh"

namespace crk {
namespace {

template <class T, int K, int B>
cudaError_t run_linear(const StepArgs& a, int wpb, cudaStream_t st) {
    const int threads = wpb * 32;
    const int grid = (a.n_strips * a.n_segs + wpb - 1) / wpb;
    StepArgs b = a;
    set_derived(b);
    bool data = false;
    for (const BCSide& s : b.bc) data = data || lin_data_side(s);
    cudaError_t e;
    if (data) {   // the boundary data first, the step as their dependent
        const dim3 faces((std::max(b.nx, b.ny) + BT_FACES - 1) / BT_FACES, 4);
        boundary_traces_kernel<T, K><<<faces, BT_FACES * (K + 1) * b.s, 0, st>>>(b);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = launch_dependent(&step2d_linear_kernel<T, K, B, true>, grid, threads, st, b);
    } else {
        step2d_linear_kernel<T, K, B, false><<<grid, threads, 0, st>>>(b);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    return launch_finalize<1>(b, st);
}

template <class T, int K, int B>
cudaError_t info_linear(KernelInfo* info) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, step2d_linear_kernel<T, K, B, false>);
    if (e != cudaSuccess) return e;
    info->regs = fa.numRegs;
    info->max_threads = fa.maxThreadsPerBlock;
    info->smem_per_thread = 0;   // the stages are combined in registers
    return cudaSuccess;
}

template <class T>
cudaError_t linear_switch(int k, int basis, const StepArgs* a, int wpb, cudaStream_t st, KernelInfo* info) {
    switch (k * 2 + (k == 0 ? 0 : basis)) {
        case 0: return a ? run_linear<T, 0, 0>(*a, wpb, st) : info_linear<T, 0, 0>(info);
        case 2: return a ? run_linear<T, 1, 0>(*a, wpb, st) : info_linear<T, 1, 0>(info);
        case 3: return a ? run_linear<T, 1, 1>(*a, wpb, st) : info_linear<T, 1, 1>(info);
        case 4: return a ? run_linear<T, 2, 0>(*a, wpb, st) : info_linear<T, 2, 0>(info);
        case 5: return a ? run_linear<T, 2, 1>(*a, wpb, st) : info_linear<T, 2, 1>(info);
        case 6: return a ? run_linear<T, 3, 0>(*a, wpb, st) : info_linear<T, 3, 0>(info);
        case 7: return a ? run_linear<T, 3, 1>(*a, wpb, st) : info_linear<T, 3, 1>(info);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_step2d_linear(int prec, int k, int basis, const StepArgs& a, int wpb, cudaStream_t st) {
    return prec == 1 ? linear_switch<double>(k, basis, &a, wpb, st, nullptr)
                     : linear_switch<float>(k, basis, &a, wpb, st, nullptr);
}

cudaError_t info_step2d_linear(int prec, int k, int basis, KernelInfo* info) {
    return prec == 1 ? linear_switch<double>(k, basis, nullptr, 0, nullptr, info)
                     : linear_switch<float>(k, basis, nullptr, 0, nullptr, info);
}

}  // namespace crk
