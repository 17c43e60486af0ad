// Fused cRKDG time step on a 2D Cartesian mesh (eq. (2.8)).
//
// Work decomposition ("marching warps"): a warp owns a strip of 30 columns
// plus one halo column on each side (lane l holds column x0 - 1 + l) and
// marches up a segment of rows.  For every row each lane
//   1. loads u^n of its cell (planes [v][m][y][x]: one coalesced 128-byte
//      line per (v, m) for the warp) and, if a limit is pending, applies the
//      TVB limiter of the previous step to it (limit-on-load);
//   2. runs every RK stage cell-locally (eq. (2.8), first line): stage states
//      u^(i) and div^loc f(u^(i)) (eq. (2.7)) stay in registers and in the
//      thread's private shared-memory slots; nothing of a stage reaches HBM;
//   3. forms the final-stage face fluxes sum_i b_i fhat(u^(i)) (eq. (2.8),
//      second line): east/west faces with the neighbouring lane through
//      warp shuffles, south faces with the north traces of the row below,
//      kept per stage in the same thread's shared-memory slot;
//   4. completes the update of the row below (its north face is the current
//      row's south face) and writes u^{n+1} of that row once.
// Halo columns are recomputed instead of exchanged: the compactness of cRKDG
// (Sec. 3.1) means one ring suffices.  So is the row beyond each end of a
// segment, two rows per segment, where rows are cheap or segments long (2 of 28
// rows on the 1920 x 480 mesh).  Elsewhere (use_seams) the faces between two
// segments (seams) are left to two small launches: a segment keeps its first
// row's south and its last row's north traces in a scratch array and the two
// rows' updates unfinished; seam_flux_kernel forms the seams' fluxes, seam_kernel
// completes the rows and ends the step.  Both ways do the same operations in the
// same order for every cell: the result does not depend on the segments, bit for
// bit.  (Completing a seam at the end of the warp that finished last, by a
// counter per row, was slower than the launches: 2.48 against 2.26 ms for two
// steps of P^2 in FP64 on 640 x 160, 2.45 against 1.82 ms for twenty of the
// deviation form on 320 x 320: each warp's end was a chain of fences, atomics and
// loads.)
// Boundary data enter only the final-stage fluxes, at t^n + c_i dt (Sec. 3.4).
// The FP64 epilogue reduces the new cell averages (max wave speed, totals;
// eq. (3.4)) per warp; the launch that ends the step (finalize_step_kernel or
// seam_kernel) combines the warps' slots and updates the device run state.
#pragma once
#include "common.cuh"
#include "launch.h"
#include "limiter.cuh"
#include "mlp_warp.cuh"

// launch bounds of the single-problem step kernel (tuning knobs)
#ifndef CRK_STEP_MAXT
#define CRK_STEP_MAXT 256
#endif
#ifndef CRK_STEP_MINB2
#define CRK_STEP_MINB2 1
#endif
// blocks per SM the scalar (advection) step is compiled for: its live state
// is a quarter of the Euler step's, so it can trade registers for warps
#ifndef CRK_STEP_MINB_ADV
#define CRK_STEP_MINB_ADV 2
#endif

namespace crk {

// a0 += x0 * c, a1 += x1 * c: one packed FP32x2 FMA on sm_100+ for float
// (the same fused rounding as two scalar FMAs), two FMAs for double
template <class T>
__device__ __forceinline__ void pfma(T& a0, T& a1, T x0, T x1, T c) {
    if constexpr (sizeof(T) == 4) {
        const float2 r = __ffma2_rn(make_float2(x0, x1), make_float2(c, c), make_float2(a0, a1));
        a0 = r.x;
        a1 = r.y;
    } else {
        a0 = fma(x0, c, a0);
        a1 = fma(x1, c, a1);
    }
}

// packed sum, difference and scaling of pairs: one FP32x2 instruction each
// on sm_100+ for float (rounding as the scalar operations), scalar for double
template <class T>
__device__ __forceinline__ void padd(T& r0, T& r1, T a0, T a1, T b0, T b1) {
    if constexpr (sizeof(T) == 4) {
        const float2 r = __fadd2_rn(make_float2(a0, a1), make_float2(b0, b1));
        r0 = r.x;
        r1 = r.y;
    } else {
        r0 = a0 + b0;
        r1 = a1 + b1;
    }
}
template <class T>
__device__ __forceinline__ void psub(T& r0, T& r1, T a0, T a1, T b0, T b1) {
    if constexpr (sizeof(T) == 4) {
        const float2 r = __ffma2_rn(make_float2(b0, b1), make_float2(-1.f, -1.f), make_float2(a0, a1));
        r0 = r.x;
        r1 = r.y;
    } else {
        r0 = a0 - b0;
        r1 = a1 - b1;
    }
}
template <class T>
__device__ __forceinline__ void pmul(T& a0, T& a1, T c) {
    if constexpr (sizeof(T) == 4) {
        const float2 r = __fmul2_rn(make_float2(a0, a1), make_float2(c, c));
        a0 = r.x;
        a1 = r.y;
    } else {
        a0 *= c;
        a1 *= c;
    }
}

template <class T, int K, int B, int PHYS>
struct Step2D {
    using TB = Tab2D<K, B>;
    static constexpr int NQ = TB::NQ;
    static constexpr int NQV = TB::NQV;
    static constexpr int NM = TB::NM;
    static constexpr int NV = Phys<T, PHYS>::NV;
    static constexpr int NDOF = NV * NM;
    static constexpr int NRED = NV + 2;   // reduction slots: maxspeed, sums[NV], troubled

    // T elements of private shared memory per thread for s stages: L_j
    // (j < s-1), north traces per stage, pending update
    static __host__ __device__ constexpr int smem_per_thread(int s) { return (s - 1) * NDOF + s * NQ * NV + NDOF; }
};

// The seam scratch of the segments, per segment and column: the first row's
// south traces (per stage), the last row's north traces, the first row's
// north-face flux (and, in deviation form, its move between the two rows' bases),
// the flux of the seam below it (likewise), its volume term and, with the limit
// on load, its limited u^n.  Values of
// entry k of all columns lie together.  (Its east/west face terms wait in the
// output buffer, as a last row's update does.)
template <class T, int K, int B, int PHYS, bool DEV>
struct Seam {
    using C = Step2D<T, K, B, PHYS>;
    static constexpr int NF = C::NQ * C::NV;
    T* base;
    size_t nx, seg_size;
    int ntr;
    __device__ __forceinline__ Seam(void* scratch, int s, int nx_, bool lim)
        : base(static_cast<T*>(scratch)), nx(nx_), seg_size(seam_values(s, C::NQ, C::NV, C::NM, DEV, lim, nx_)),
          ntr(s * NF) {}
    __device__ __forceinline__ T* at(int seg, int k, int col) const { return base + seg * seg_size + k * nx + col; }
    __device__ __forceinline__ T* south(int seg, int k, int col) const { return at(seg, k, col); }
    __device__ __forceinline__ T* north(int seg, int k, int col) const { return at(seg, ntr + k, col); }
    __device__ __forceinline__ T* flux(int seg, int k, int col) const { return at(seg, 2 * ntr + k, col); }
    // the flux of the seam below the segment (and its move between bases)
    __device__ __forceinline__ T* below(int seg, int k, int col) const {
        return at(seg, 2 * ntr + NF + (DEV ? C::NV : 0) + k, col);
    }
    __device__ __forceinline__ T* vol(int seg, int k, int col) const {
        return at(seg, 2 * (ntr + NF + (DEV ? C::NV : 0)) + k, col);
    }
    __device__ __forceinline__ T* un(int seg, int k, int col) const {
        return at(seg, 2 * (ntr + NF + (DEV ? C::NV : 0)) + C::NDOF + k, col);
    }
};

// First row of segment seg of nseg (rows split evenly); the 64-bit division
// only where the product needs it
__device__ __forceinline__ int seg_row(int seg, int ny, int nseg) {
    const unsigned long long n = (unsigned long long)seg * ny;
    return n >> 32 ? (int)(n / nseg) : (int)((unsigned)n / (unsigned)nseg);
}

// Per-problem view of one step.  The single-problem kernel reads the mesh
// straight from its launch arguments (kernel-parameter constant bank, no
// registers held); the batched kernel reads it from the problem table.
template <class T>
struct ArgsView {
    const StepArgs& a;
    double t_, dt_;
    __device__ __forceinline__ const T* uin() const { return static_cast<const T*>(a.uin); }
    __device__ __forceinline__ T* uout() const { return static_cast<T*>(a.uout); }
    __device__ __forceinline__ int nx() const { return a.nx; }
    __device__ __forceinline__ int ny() const { return a.ny; }
    __device__ __forceinline__ double x0() const { return a.x0; }
    __device__ __forceinline__ double y0() const { return a.y0; }
    __device__ __forceinline__ double dx() const { return a.dx; }
    __device__ __forceinline__ double dy() const { return a.dy; }
    __device__ __forceinline__ double t() const { return t_; }
    __device__ __forceinline__ double dt() const { return dt_; }
    __device__ __forceinline__ int n_strips() const { return a.n_strips; }
    __device__ __forceinline__ int n_segs() const { return a.n_segs; }
    __device__ __forceinline__ int total_warps() const { return a.n_strips * a.n_segs; }
    __device__ __forceinline__ double* partials() const { return a.partials; }
    __device__ __forceinline__ void* seam() const { return a.seam; }
    __device__ __forceinline__ DevState* ds() const { return a.ds; }
    __device__ __forceinline__ int* cur() const { return nullptr; }
    __device__ __forceinline__ unsigned* done() const { return nullptr; }
    static constexpr bool ALONE = true;   // the one problem of its launch
    __device__ __forceinline__ bool copy_if_idle() const { return true; }
    // derived constants, computed on the host (set_derived)
    __device__ __forceinline__ T rxT() const {
        if constexpr (sizeof(T) == 4) return a.rxf;
        else return T(a.rx);
    }
    __device__ __forceinline__ T ryT() const {
        if constexpr (sizeof(T) == 4) return a.ryf;
        else return T(a.ry);
    }
    __device__ __forceinline__ T Mdx2T() const {
        if constexpr (sizeof(T) == 4) return a.Mdx2f;
        else return T(a.M * a.dx * a.dx);
    }
    __device__ __forceinline__ T Mdy2T() const {
        if constexpr (sizeof(T) == 4) return a.Mdy2f;
        else return T(a.M * a.dy * a.dy);
    }
    __device__ __forceinline__ double cell() const { return a.cell; }
    __device__ __forceinline__ double adv_speed() const { return a.adv_speed; }
};

template <class T>
struct ProbView {
    const T* uin_;
    T* uout_;
    int nx_, ny_;
    double x0_, y0_, dx_, dy_;
    double t_, dt_;
    int n_strips_, n_segs_, total_warps_;
    double* partials_;    // this problem's reduction slots
    void* seam_;          // this problem's seam scratch
    DevState* ds_;        // this problem's run state
    int* cur_;            // this problem's buffer index (flipped at the end of its step)
    unsigned* done_;      // count of problems that reached t_end
    __device__ __forceinline__ const T* uin() const { return uin_; }
    __device__ __forceinline__ T* uout() const { return uout_; }
    __device__ __forceinline__ int nx() const { return nx_; }
    __device__ __forceinline__ int ny() const { return ny_; }
    __device__ __forceinline__ double x0() const { return x0_; }
    __device__ __forceinline__ double y0() const { return y0_; }
    __device__ __forceinline__ double dx() const { return dx_; }
    __device__ __forceinline__ double dy() const { return dy_; }
    __device__ __forceinline__ double t() const { return t_; }
    __device__ __forceinline__ double dt() const { return dt_; }
    __device__ __forceinline__ int n_strips() const { return n_strips_; }
    __device__ __forceinline__ int n_segs() const { return n_segs_; }
    __device__ __forceinline__ int total_warps() const { return total_warps_; }
    __device__ __forceinline__ double* partials() const { return partials_; }
    __device__ __forceinline__ void* seam() const { return seam_; }
    __device__ __forceinline__ DevState* ds() const { return ds_; }
    __device__ __forceinline__ int* cur() const { return cur_; }
    __device__ __forceinline__ unsigned* done() const { return done_; }
    static constexpr bool ALONE = false;
    __device__ __forceinline__ bool copy_if_idle() const { return false; }
    // per-problem constants, in the arithmetic of set_derived (1/dx and 1/dy
    // from the problem table, made on the host)
    double rx_, ry_, M_, bx_, by_;
    __device__ __forceinline__ T rxT() const { return T(rx_); }
    __device__ __forceinline__ T ryT() const { return T(ry_); }
    __device__ __forceinline__ T Mdx2T() const { return T(M_ * dx_ * dx_); }
    __device__ __forceinline__ T Mdy2T() const { return T(M_ * dy_ * dy_); }
    __device__ __forceinline__ double cell() const { return dx_ * dy_; }
    __device__ __forceinline__ double adv_speed() const { return fabs(bx_) / dx_ + fabs(by_) / dy_; }
};

// Device run-state update after a step from the reduced slots: t, the next
// dt = min(cfl / max speed, t_end - t), totals, troubled count.
// cfl, t_end, lim_count: the run state's values (not written by the step)
__device__ __forceinline__ void finish_run_state(const StepArgs& a, DevState* ds, double mx, const double* sm_,
                                                 int nv, double tr, double t0, double dt, double cfl,
                                                 double t_end, unsigned long long lim_count, int* cur,
                                                 unsigned* done) {
    ds->maxspeed = mx;
    for (int v = 0; v < nv; ++v) ds->sums[v] = sm_[v];
    // troubled cells: this step's limit-on-load, else a separate pass over u^n
    ds->troubled = a.limit ? tr : double(lim_count);
    ds->lim_count = 0;
    const double tn = t0 + dt;
    ds->t = tn;
    double dn = cfl > 0.0 && mx > 0.0 ? cfl / mx : dt;
    const double rem = t_end - tn;
    const bool reached = rem <= 1e-12 * fmax(1.0, fabs(t_end));
    if (dn > rem) dn = rem;
    if (reached) dn = 0.0;
    ds->dt = dn;
    ds->steps += 1;
    ds->counter = 0;
    if (cur) *cur ^= 1;
    if (done && reached) atomicAdd(done, 1u);
}

// NV values summed over a warp's lanes (every lane returns lane v's sum of
// value v, v < NV): the lanes of a pair each take over half of the values, so
// four FP64 sums need 6 additions a lane instead of 20 (FP64 runs at 1/64 of
// the FP32 rate).
template <int NV>
__device__ __forceinline__ void warp_sums(double (&v)[NV]) {
    const int lane = threadIdx.x & 31;
    constexpr unsigned ALL = 0xffffffffu;
    if constexpr (NV == 4) {
        const bool h = lane & 16, q = lane & 8;
        const double a0 = (h ? v[2] : v[0]) + __shfl_xor_sync(ALL, h ? v[0] : v[2], 16);
        const double a1 = (h ? v[3] : v[1]) + __shfl_xor_sync(ALL, h ? v[1] : v[3], 16);
        double x = (q ? a1 : a0) + __shfl_xor_sync(ALL, q ? a0 : a1, 8);
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) x += __shfl_xor_sync(ALL, x, off);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = __shfl_sync(ALL, x, 8 * i);
    } else {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
            for (int i = 0; i < NV; ++i) v[i] += __shfl_xor_sync(ALL, v[i], off);
    }
}

// FP64 epilogue of a step: warp reduction of the lane accumulators (max
// wave speed, NV totals, troubled count, status bits) into the warp's slot
// (NV + 2 doubles; the totals without the cell's area, the maximum as an
// ordered key, the count as an integer, both stored bitwise).  The launch that
// follows the step reduces the slots.
template <int NV, int NRED, class PV>
__device__ __forceinline__ void step_epilogue(const PV& pv, int gw, int lane, double red_max, double (&red_sum)[NV],
                                              unsigned red_trouble, unsigned status) {
    static_assert(NRED == NV + 2, "slot layout: max speed, NV totals, troubled count");
    unsigned long long key = speed_key(red_max);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long k = __shfl_xor_sync(0xffffffffu, key, off);
        key = k > key ? k : key;
    }
    warp_sums<NV>(red_sum);
    red_trouble = __reduce_add_sync(0xffffffffu, red_trouble);
    status = __reduce_or_sync(0xffffffffu, status);
    if (lane == 0) {
        double* slotp = pv.partials() + (size_t)gw * NRED;
        slotp[0] = __longlong_as_double((long long)key);
#pragma unroll
        for (int v = 0; v < NV; ++v) slotp[1 + v] = red_sum[v];
        slotp[1 + NV] = __longlong_as_double((long long)red_trouble);
        if (status) atomicOr(&pv.ds()->status, status);
    }
}

// What a block holds of the reductions, and the sum over its threads (fixed
// order: deterministic); thread 0 holds the result.
template <int NV>
struct StepRed {
    unsigned long long key = 0, trouble = 0;
    double sum[NV] = {};
    __device__ __forceinline__ void add_slot(const double* q) {
        double e[NV + 2];
#pragma unroll
        for (int i = 0; i < NV + 2; ++i) e[i] = __ldcg(q + i);
        const unsigned long long k = (unsigned long long)__double_as_longlong(e[0]);
        key = k > key ? k : key;
#pragma unroll
        for (int v = 0; v < NV; ++v) sum[v] += e[1 + v];
        trouble += (unsigned long long)__double_as_longlong(e[1 + NV]);
    }
    __device__ __forceinline__ void put_slot(double* q) const {
        q[0] = __longlong_as_double((long long)key);
#pragma unroll
        for (int v = 0; v < NV; ++v) q[1 + v] = sum[v];
        q[1 + NV] = __longlong_as_double((long long)trouble);
    }
    __device__ __forceinline__ void warp_reduce() {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long k = __shfl_xor_sync(0xffffffffu, key, off);
            key = k > key ? k : key;
            trouble += __shfl_xor_sync(0xffffffffu, trouble, off);
        }
        warp_sums<NV>(sum);
    }
    template <int NT>
    __device__ __forceinline__ void block_reduce() {
        warp_reduce();
        if constexpr (NT > 32) {
            constexpr int NW = NT / 32;
            __shared__ double slots[NW][NV + 2];
            const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
            __syncthreads();   // an earlier call's slots have been read
            if (lane == 0) put_slot(slots[w]);
            __syncthreads();
            if (threadIdx.x == 0)
#pragma unroll
                for (int i = 1; i < NW; ++i) {
                    const unsigned long long k = (unsigned long long)__double_as_longlong(slots[i][0]);
                    key = k > key ? k : key;
#pragma unroll
                    for (int v = 0; v < NV; ++v) sum[v] += slots[i][1 + v];
                    trouble += (unsigned long long)__double_as_longlong(slots[i][1 + NV]);
                }
        }
    }
};

// A step kernel's follow-up launch as its programmatic dependent: the step's
// blocks allow it early (griddepcontrol.launch_dependents), so its blocks are
// scheduled as soon as an SM has room and wait for the step's completion,
// without a launch gap
template <class... A, class... V>
inline cudaError_t launch_dependent(void (*kern)(A...), int grid, int threads, cudaStream_t st, V... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, A(args)...);
}
// ... which waits here until the step grid has completed and its writes are visible
__device__ __forceinline__ void wait_for_step() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The end of a single-problem step without seams, as its own launch of one block: each
// thread reduces a run of slots, then fixed-order trees; thread 0 updates the
// device run state.  A last warp of the step itself would reduce ~1,000-2,400
// slots alone while the rest of the GPU idles.
constexpr int FINALIZE_THREADS = 256;

template <int NV>
__global__ void __launch_bounds__(FINALIZE_THREADS) finalize_step_kernel(const StepArgs a, int total_warps) {
    wait_for_step();
    DevState* ds = a.ds;
    const double dt = a.dt_from_dev ? ds->dt : a.dt;
    if (!(dt > 0.0)) return;   // the step left the state and the run state unchanged
    StepRed<NV> red;
#pragma unroll 4
    for (int w = threadIdx.x; w < total_warps; w += FINALIZE_THREADS)
        red.add_slot(a.partials + (size_t)w * (NV + 2));
    red.template block_reduce<FINALIZE_THREADS>();
    if (threadIdx.x == 0) {
        for (int v = 0; v < NV; ++v) red.sum[v] *= a.cell;
        finish_run_state(a, ds, __longlong_as_double((long long)red.key), red.sum, NV, double(red.trouble),
                         a.dt_from_dev ? ds->t : a.t, dt, ds->cfl, ds->t_end, ds->lim_count, nullptr, nullptr);
    }
}

template <int NV>
inline cudaError_t launch_finalize(const StepArgs& b, cudaStream_t st) {
    return launch_dependent(&finalize_step_kernel<NV>, 1, FINALIZE_THREADS, st, b, b.n_strips * b.n_segs);
}

// In a step kernel: its dependent finalize launch may be scheduled now
__device__ __forceinline__ void allow_dependent_launch() { asm volatile("griddepcontrol.launch_dependents;"); }

// The accumulators of the new averages' reductions: FP32 states (plain or
// compensated) keep the maximum in FP32 (GB300's FP64 pipe is 1/64 of its FP32
// rate) and the totals in compensated FP32 (TwoSum; a compensated state adds
// its lo parts into the error term), converted to FP64 once per warp; FP64
// states keep FP64.
template <class T, int NV>
struct CellRed {
    T hi[NV] = {}, lo[NV] = {};   // FP32: totals and their error terms
    T maxT = T(0);
    double max = 0.0;
    double sum[NV] = {};          // FP64
    unsigned status = 0;
    // FP64 maximum and totals (adv_speed: the one speed of a linear flux, 0 where no cell was written)
    template <int PHYS>
    __device__ __forceinline__ void close(double adv_speed) {
        if constexpr (sizeof(T) == 4) {
            max = PHYS == PHYS_EULER ? double(maxT) : adv_speed;
#pragma unroll
            for (int v = 0; v < NV; ++v) sum[v] = double(hi[v]) + double(lo[v]);
        }
    }
};

// Wave speed of new averages A, in the state's arithmetic, and its status bits
template <class T, int PHYS, int NV, class PV, class AV>
__device__ __forceinline__ T new_speed(const StepArgs& a, const PV& pv, const AV& A, T rx, T ry, T gm1, T gam,
                                       unsigned& status) {
    if constexpr (PHYS != PHYS_EULER) {
        if (!(A(0) == A(0))) status |= ST_NAN;
        return T(pv.adv_speed());
    } else {
        const T ir = T(1) / A(0);
        const T w = A(1) * ir, vv = A(2) * ir;
        const T p = gm1 * (A(3) - T(0.5) * (A(1) * w + A(2) * vv));
        const T c = sqrt(fmax(gam * p * ir, T(0)));
        T sp;
        if constexpr (sizeof(T) == 4) sp = (fabs(w) + c) * rx + (fabs(vv) + c) * ry;
        else sp = (fabs(w) + c) / pv.dx() + (fabs(vv) + c) / pv.dy();
        if (!(A(0) > T(0)) || !(p > T(0))) status |= ST_NONPHYSICAL;
        if (!(sp == sp)) status |= ST_NAN;
        return sp;
    }
}

// hi' + lo' = hi + lo + inc at element ix of a compensated state (TwoSum).  u^n
// is read through the read-only path: as ordinary loads the modes' hi and lo
// waited for one another's stores (the compiler does not see across this
// function that uout is another buffer), 72 round trips a row for Q^2.
template <class T>
__device__ __forceinline__ void store_comp(const T* __restrict__ uin, T* __restrict__ uout, size_t ix, size_t lo_off,
                                           T inc, T& hi_out, T& lo_out) {
    const T hi = __ldg(uin + ix), lo = __ldg(uin + lo_off + ix);
    const T d = inc + lo;
    const T sum = hi + d;
    const T bv = sum - hi;
    const T err = (hi - (sum - bv)) + (d - bv);
    uout[ix] = sum;
    uout[lo_off + ix] = err;
    hi_out = sum;
    lo_out = err;
}

// u^{n+1} of a cell from its finished update P (COMP: the increment, added to
// hi + lo; P[v][0] becomes the new hi average) and its part of the reductions
template <class T, int PHYS, int NV, int NM, bool COMP, class PV>
__device__ __forceinline__ void store_cell(const StepArgs& a, const PV& pv, const T* __restrict__ uin,
                                           T* __restrict__ uout, size_t plane, size_t o, T (&P)[NV][NM], T rx, T ry,
                                           T gm1, T gam, CellRed<T, NV>& red) {
    static_assert(!COMP || sizeof(T) == 4, "the compensated state is FP32");
    T avl[NV];   // COMP: lo parts of the new averages
#pragma unroll
    for (int v = 0; v < NV; ++v) {
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const size_t ix = (size_t)(v * NM + m) * plane + o;
            if constexpr (COMP) {
                T hi, lo;
                store_comp(uin, uout, ix, (size_t)(NV * NM) * plane, P[v][m], hi, lo);
                if (m == 0) {
                    P[v][0] = hi;
                    avl[v] = lo;
                }
            } else {
                uout[ix] = P[v][m];
            }
        }
    }
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {   // TwoSum: hi + lo += A[v] exactly
            const T x = P[v][0];
            const T sum = red.hi[v] + x;
            const T bv = sum - red.hi[v];
            red.lo[v] += (red.hi[v] - (sum - bv)) + (x - bv);
            if constexpr (COMP) red.lo[v] += avl[v];
            red.hi[v] = sum;
        }
        const T sp = new_speed<T, PHYS, NV>(a, pv, [&](int v) { return P[v][0]; }, rx, ry, gm1, gam, red.status);
        if constexpr (PHYS == PHYS_EULER) red.maxT = fmax(red.maxT, sp);
    } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) red.sum[v] += P[v][0];
        red.max = fmax(red.max, new_speed<T, PHYS, NV>(a, pv, [&](int v) { return P[v][0]; }, rx, ry, gm1, gam, red.status));
    }
}

// One variable's update of a row in two parts, the same operations wherever a
// row is completed.  First: sx the east/west face terms, V the volume term, FS the
// flux of the south face; P = u^n (COMP: 0) minus dt times the operator without
// its north face.
template <class T, int K, int B, bool COMP, bool SQ, int NQ, int NM>
__device__ __forceinline__ void row_update(T (&P)[NM], const T (&sx)[NM], const T (&V)[NM], const T (&FS)[NQ],
                                           const T (&un)[NM], T rx, T ry, T tdt) {
    static_for<NM>([&](auto mc) {
        constexpr int m = decltype(mc)::value;
        T sy = T(0);
        static_for<NQ>([&](auto pc) {
            constexpr double w = Const2D<K, B>::tab.pS[decltype(pc)::value][m];
            if constexpr (w != 0.0) sy = fma(FS[decltype(pc)::value], T(-w), sy);
        });
        const T fsum = SQ ? fma(rx, sx[m] + sy, -V[m]) : fma(rx, sx[m], ry * sy) - V[m];
        constexpr double cm = Const2D<K, B>::tab.cm[m];
        const T tc = tdt * T(cm);
        if constexpr (COMP) P[m] = -tc * fsum;
        else P[m] = fma(-tc, fsum, un[m]);
    });
}
// ... and the north face: FN its flux (DEV: relative to the base of the row
// above, gS moves it to this row's)
template <class T, int K, int B, bool DEV, int NQ, int NM>
__device__ __forceinline__ void add_north(T (&P)[NM], const T (&FN)[NQ], T gS, T ry, T tdt) {
    static_for<NM>([&](auto mc) {
        constexpr int m = decltype(mc)::value;
        T s = T(0);
        static_for<NQ>([&](auto pc) {
            constexpr double w = Const2D<K, B>::tab.pN[decltype(pc)::value][m];
            if constexpr (w != 0.0) s = fma(FN[decltype(pc)::value], T(w), s);
        });
        constexpr double sN = Const2D<K, B>::tab.sN[m], cm = Const2D<K, B>::tab.cm[m];
        if constexpr (DEV && sN != 0.0) s = fma(gS, T(-sN), s);
        P[m] = fma(-(tdt * T(cm)), ry * s, P[m]);
    });
}
template <int NQ, int NV, class T>
__device__ __forceinline__ void column(const T (&F)[NQ][NV], int v, T (&out)[NQ]) {
#pragma unroll
    for (int p = 0; p < NQ; ++p) out[p] = F[p][v];
}

// COMP = true: compensated FP32 state.  The buffers hold hi planes followed
// by lo planes (u = hi + lo); every stage computes in T from hi, and only the
// final update u^{n+1} = u^n + Delta is accumulated exactly (TwoSum of hi and
// Delta + lo), so the state does not collect one rounding of its own size
// per step.  Used without limiters.
// MLPI = true: the troubled-cell decision of the limit-on-load comes from the
// learned indicator (BF16 tensor-core MLP over the warp's 32 cells): limit if
// the logit exceeds mlp_zhi, keep if it is below mlp_zlo, and let the TVB test
// decide in between.  The weights sit in shared memory after the threads'
// private slots, followed by one staging area per warp.
template <class T, int K, int B, int PHYS>
__host__ __device__ constexpr size_t mlp_smem_offset(int s, int nthr) {
    return ((size_t)Step2D<T, K, B, PHYS>::smem_per_thread(s) * sizeof(T) * nthr + 15) / 16 * 16;
}
constexpr size_t mlp_smem_bytes(int nthr) {
    return sizeof(MlpSmem) + (size_t)(nthr / 32) * (32 * MLP_INP + 64) * sizeof(__nv_bfloat16);
}

// LIM = false: an instantiation without the limit-on-load code, for steps
// whose u^n needs no limiting here (none pending, or a separate pass did it).
// DEV = true (with COMP, 2D Euler, FP32): every state is held as its
// deviation from the cell's base state (the high part of its average at t^n)
// and every flux in deviation form (EulerDev), so that the stage operators
// and the final stage carry FP32 errors relative to their own size; the
// compensated state then accumulates increments that are accurate to a few
// ulps of themselves.  Face traces and face fluxes that cross to a
// neighbouring cell move to its base by the deviation of the base
// difference.  Inner stages, final stage and the update all run on the FP32
// pipe.
// SQ = true (square cells, dx == dy, so 1/dx == 1/dy): the face terms
// accumulate without the 1/dx factors, applied once to each local-operator
// value and to the update (rx (sx + sy) - V for rx sx + ry sy - V): 4 packed
// multiplications per face point fewer.
// SEAM = true: the faces between segments are left to the seam launches;
// false: the row beyond each end of the segment is recomputed instead.
template <class T, int K, int B, int PHYS, bool COMP, bool MLPI, bool LIM, bool DEV, bool SQ, bool SEAM, class PV>
__device__ __forceinline__ void step2d_body(const StepArgs& a, const PV& pv, const int gw) {
    static_assert(!DEV || (COMP && PHYS == PHYS_EULER && sizeof(T) == 4 && !MLPI && !LIM),
                  "the deviation form is built for the compensated FP32 2D Euler step without limiters");
    using C = Step2D<T, K, B, PHYS>;
    using TBL = typename C::TB;
    constexpr int NQ = C::NQ, NQV = C::NQV, NM = C::NM, NV = C::NV;
    constexpr TBL tb = make_tab2d<K, B>();

    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    const int nthr = blockDim.x;
    const int tid = threadIdx.x;
    const int S = a.s;
    const int offN = (S - 1) * C::NDOF;
    const int offP = offN + S * NQ * NV;
    // the thread's private slots: its warp holds smem_per_thread(S) rows of
    // 32 values, one column per lane (consecutive lanes in consecutive banks),
    // so that slot k sits k * 32 values past the thread's own base
    T* const smt = sm + (size_t)(tid >> 5) * (C::smem_per_thread(S) * 32) + (tid & 31);
    auto slot = [&](int k) -> T& { return smt[k * 32]; };

    const int lane = tid & 31;
    const int nx = pv.nx(), ny = pv.ny();
    const size_t plane = (size_t)nx * ny;
    const T* __restrict__ uin = pv.uin();
    T* __restrict__ uout = pv.uout();

    const double dt = pv.dt();
    const double t0 = pv.t();

    const int strip = gw % pv.n_strips();
    const int seg = gw / pv.n_strips();
    const int xs = strip * 30;
    const int col = xs - 1 + lane;
    const bool perx = a.bc[0].type == BC_PERIODIC;
    const bool pery = a.bc[2].type == BC_PERIODIC;
    int xl = ((col % nx) + nx) % nx;
    if (!perx) xl = col < 0 ? 0 : (col >= nx ? nx - 1 : col);
    const bool outlane = lane >= 1 && lane <= 30 && col < nx;
    const bool has_bcW = !perx && xs == 0;
    const bool has_bcE = !perx && xs + 30 >= nx;

    // rows split evenly over the segments.  (Either form gives the same rows, as
    // either form of keep_north's first condition below is the same condition:
    // the choice moves the compiler's schedule of the whole row.  Halo rows, FP32,
    // times over the other forms: Q^1 SSP-RK3 on 1280^2 0.971, P^2 0.989, Q^2 RK4
    // 0.996; the deviation form and a batch's kernels, which hold two bodies, keep
    // the other condition: 0.966 for the deviation form's Q^2 RK4.)
    int r0, r1;
    if constexpr (SEAM || !PV::ALONE) {
        r0 = seg_row(seg, ny, pv.n_segs());
        r1 = seg_row(seg + 1, ny, pv.n_segs());
    } else {
        r0 = (int)(((long long)seg * ny) / pv.n_segs());
        r1 = (int)(((long long)(seg + 1) * ny) / pv.n_segs());
    }
    // the faces below the first and above the last row that are seams, or the
    // halo rows that are recomputed for them
    const bool seamS = SEAM && (r0 > 0 || pery), seamN = SEAM && (r1 < ny || pery);
    const int rstart = !SEAM && (r0 > 0 || pery) ? r0 - 1 : r0;
    const int rend = !SEAM && (r1 < ny || pery) ? r1 : r1 - 1;

    // a non-positive dt leaves the state unchanged (runs past t_end)
    if (!(dt > 0.0)) {
        if (pv.copy_if_idle() && outlane)
            for (int r = r0; r < r1; ++r)
                for (int d = 0; d < (COMP ? 2 : 1) * C::NDOF; ++d)
                    uout[d * plane + (size_t)r * nx + col] = uin[d * plane + (size_t)r * nx + col];
        return;
    }

    // launch constants: 1/dx, 1/dy and the limiter thresholds made on the host
    // (set_derived), no FP64 division per warp
    constexpr bool F32 = sizeof(T) == 4;
    std::conditional_t<DEV, EulerDev<T>, Phys<T, PHYS>> ph;
    if constexpr (PHYS == PHYS_EULER) {
        ph.gamma = T(a.gamma);
        ph.gm1 = T(a.gamma - 1.0);
    } else {
        ph.bx = T(a.beta[0]);
        ph.by = T(a.beta[1]);
    }
    const T rx = opaque(pv.rxT()), ry = opaque(pv.ryT());   // held in registers, as when computed
    // the factors of the face terms (SQ: 1, applied later); the volume
    // term keeps its factors, whose products also form the register pairs of
    // its packed accumulation
    const T rxv = SQ ? T(1) : rx, ryv = SQ ? T(1) : ry;
    const T tdt = T(dt);
    const T Mdx2 = pv.Mdx2T(), Mdy2 = pv.Mdy2T();
    const T gam = T(a.gamma), gm1 = T(a.gamma - 1.0);
    const bool do_tvb = a.tvb_on, do_pp = a.pp_on;
    const T pp_eps = F32 ? T(a.pp_epsf) : T(a.pp_eps);

    const double adv_speed = PHYS == PHYS_EULER ? 0.0 : pv.adv_speed();
    CellRed<T, NV> red;
    unsigned red_trouble = 0;
    const Seam<T, K, B, PHYS, DEV> sc(pv.seam(), S, nx, LIM && a.limit);

    // limiter: rolling neighbour averages of this column
    T avg_prev[NV], avg_next[NV];
    auto load_avg = [&](int r, T* out) {
        // average of (column xl, row r), r in [-1, ny]; beyond a non-periodic
        // side: ghost average from the boundary cell (at time t^n)
        int rr = r;
        bool ghost = false;
        if (r < 0) { if (pery) rr = r + ny; else { rr = 0; ghost = true; } }
        if (r >= ny) { if (pery) rr = r - ny; else { rr = ny - 1; ghost = true; } }
        T own[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) own[v] = uin[(size_t)(v * NM) * plane + (size_t)rr * nx + xl];
        if (!ghost) {
#pragma unroll
            for (int v = 0; v < NV; ++v) out[v] = own[v];
        } else {
            cold_branch();
            const int side = r < 0 ? 2 : 3;
            const int colc = opaque(col);
            bc_exterior<T, NV>(a.bc[side], 1, own, [&](double& x, double& y, double& t) {
                x = pv.x0() + (colc + 0.5) * pv.dx();
                y = r < 0 ? pv.y0() - 0.5 * pv.dy() : pv.y0() + (ny + 0.5) * pv.dy();
                t = t0;
            }, out);
        }
    };
    auto load_avg_x = [&](int c, int r, T* out) {
        // average of column c (may be -1 .. nx) in row r (0..ny-1)
        T own[NV];
        int cc = perx ? ((c % nx) + nx) % nx : (c < 0 ? 0 : (c >= nx ? nx - 1 : c));
#pragma unroll
        for (int v = 0; v < NV; ++v) own[v] = uin[(size_t)(v * NM) * plane + (size_t)r * nx + cc];
        if (perx || (c >= 0 && c < nx)) {
#pragma unroll
            for (int v = 0; v < NV; ++v) out[v] = own[v];
        } else {
            cold_branch();
            const int side = c < 0 ? 0 : 1;
            const int rc = opaque(r);
            bc_exterior<T, NV>(a.bc[side], 0, own, [&](double& x, double& y, double& t) {
                x = c < 0 ? pv.x0() - 0.5 * pv.dx() : pv.x0() + (nx + 0.5) * pv.dx();
                y = pv.y0() + (rc + 0.5) * pv.dy();
                t = t0;
            }, out);
        }
    };
    if (LIM && a.limit) load_avg(rstart - 1, avg_prev);
    T cprev[NV];   // DEV: base state of the row below (the previous row of the march)
#pragma unroll
    for (int v = 0; v < NV; ++v) cprev[v] = T(0);
    const double hh_ = pv.dx() > pv.dy() ? pv.dx() : pv.dy();
    const double mlp_scale = a.M * hh_ * hh_;

    for (int r = rstart; r <= rend; ++r) {
        const int ry_ = SEAM ? r : (r < 0 ? r + ny : (r >= ny ? r - ny : r));
        const bool out_row = SEAM || (r >= r0 && r < r1);
        const bool south_bc = (r == 0) && !pery;
        const bool do_south = r > rstart || south_bc;   // flux through this row's south face
        const bool seam_row = SEAM && r == r0 && seamS; // its update waits for the seam below it
        const bool last = r == rend;
        const bool keep_north = SEAM ? !last || !seamN : ((DEV || !PV::ALONE ? !last : r < rend) || (r == ny - 1 && !pery && out_row));

        // ---- load u^n (and limit on load) -------------------------------------
        T un[NV][NM];
        const size_t cidx = (size_t)ry_ * nx + xl;
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int m = 0; m < NM; ++m) un[v][m] = uin[(size_t)(v * NM + m) * plane + cidx];

        // DEV: the base cb = hi part of the average; un becomes the deviation
        // (lo of the average, hi + lo of the higher modes); cS is the base of
        // the row below.  The neighbours' bases minus this cell's are formed
        // where they are used (fewer live registers)
        T cb[NV], cS[NV];
        if constexpr (DEV) {
            const size_t lo_off = (size_t)C::NDOF * plane;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                cb[v] = un[v][0];
                un[v][0] = uin[lo_off + (size_t)(v * NM) * plane + cidx];
#pragma unroll
                for (int m = 1; m < NM; ++m) un[v][m] += uin[lo_off + (size_t)(v * NM + m) * plane + cidx];
            }
            ph.set_base(cb);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                cS[v] = cprev[v];
                cprev[v] = cb[v];
            }
        }
        // exterior state at a boundary point from an interior trace (DEV:
        // both as deviations from this cell's base; the affine sides exactly)
        auto bcx = [&](const BCSide& bc, int axis, const T* din, auto&& xyt, T* out) {
            if constexpr (DEV) {
                if (bc.affine) {
#pragma unroll
                    for (int v = 0; v < NV; ++v)
                        out[v] = fma(T(bc.m[v]), din[v], fma(T(bc.m[v]) - T(1), cb[v], T(bc.cf[v])));
                } else {
                    T full[NV];
#pragma unroll
                    for (int v = 0; v < NV; ++v) full[v] = cb[v] + din[v];
                    bc_exterior<T, NV>(bc, axis, full, xyt, out);
#pragma unroll
                    for (int v = 0; v < NV; ++v) out[v] -= cb[v];
                }
            } else {
                bc_exterior<T, NV>(bc, axis, din, xyt, out);
            }
        };

        if (LIM && a.limit) {
            T avg_cur[NV], nbW[NV], nbE[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) avg_cur[v] = un[v][0];
            load_avg(r + 1, avg_next);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                nbE[v] = shfl_down(avg_cur[v], 1);
                nbW[v] = shfl_up(avg_cur[v], 1);
            }
            if (lane == 0) load_avg_x(col - 1, ry_, nbW);
            if (lane == 31) load_avg_x(col + 1, ry_, nbE);
            if (!perx && col == 0) load_avg_x(-1, ry_, nbW);
            if (!perx && col == nx - 1) load_avg_x(nx, ry_, nbE);
            const bool real = perx ? true : (col >= 0 && col < nx);
            bool fl = false;
            int mode = -1;
            if constexpr (MLPI) {
                // every lane takes part in the warp's MLP evaluation
                unsigned char* base = smem_raw + mlp_smem_offset<T, K, B, PHYS>(S, nthr);
                const MlpSmem& mw = *reinterpret_cast<const MlpSmem*>(base);
                __nv_bfloat16* stage = reinterpret_cast<__nv_bfloat16*>(base + sizeof(MlpSmem)) +
                                       (tid >> 5) * (32 * MLP_INP + 64);
                float feat[MLP_IN];
                mlp_features<T, NM>(un, nbE, nbW, avg_next, avg_prev, mlp_scale, feat);
                const float z = mlp_warp_logit(mw, feat, stage);
                mode = z > a.mlp_zhi ? 1 : (z < a.mlp_zlo ? 0 : -1);
            }
            if (real && do_tvb)
                fl = tvb_limit_cell<T, NV, NM>(un, nbW, nbE, avg_prev, avg_next, Mdx2, Mdy2, gam, mode);
            if (real && do_pp) positivity_cell<T, NV, NM, K, B>(un, gam, pp_eps);
            if (out_row && outlane && fl) ++red_trouble;
#pragma unroll
            for (int v = 0; v < NV; ++v) avg_prev[v] = avg_cur[v];
        }

        // ---- stages ---------------------------------------------------------------
        T V[NV][NM];      // sum_i b_i * volume term
        T FE[NQ][NV];     // sum_i b_i fhat on the east face
        T FS[NQ][NV];     // sum_i b_i fhat on the south face
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int m = 0; m < NM; ++m) V[v][m] = T(0);
#pragma unroll
        for (int p = 0; p < NQ; ++p)
#pragma unroll
            for (int v = 0; v < NV; ++v) FE[p][v] = FS[p][v] = T(0);

        for (int i = 0; i < S; ++i) {
            const T bi = tab_bT<T>(a, i);
            const T hbi = T(0.5) * bi;   // the weight of the east and south fluxes formed without their 1/2
            const bool need_L = i < S - 1;
            const bool need_flux = bi != T(0);
            if (!need_L && !need_flux) continue;
            // stage state u^(i) = u^n - dt sum_{j<i} a_ij L_j
            T w[NV][NM];
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int m = 0; m < NM; ++m) w[v][m] = un[v][m];
            for (int j = 0; j < i; ++j) {
                const T aijT = tab_aT<T>(a, i, j);
                if (aijT == T(0)) continue;
                const T aij = aijT * tdt;
                if constexpr (NV % 2 == 0) {
#pragma unroll
                    for (int v = 0; v < NV; v += 2)
#pragma unroll
                        for (int m = 0; m < NM; ++m)
                            pfma(w[v][m], w[v + 1][m], slot(j * C::NDOF + v * NM + m),
                                 slot(j * C::NDOF + (v + 1) * NM + m), -aij);
                } else {
#pragma unroll
                    for (int v = 0; v < NV; ++v)
#pragma unroll
                        for (int m = 0; m < NM; ++m) w[v][m] -= aij * slot(j * C::NDOF + v * NM + m);
                }
            }
            // volume term  sum_q w_q (rx f_x dphi/dxi + ry f_y dphi/deta)
            T vol[NV][NM];
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int m = 0; m < NM; ++m) vol[v][m] = T(0);
            // flux and projection of the point values uq at volume point q
            auto vol_point = [&](const int q, const T (&uq)[NV]) {
                T fx[NV], fy[NV];
                ph.flux2(uq, fx, fy);
                if constexpr (NV % 2 == 0) {
#pragma unroll
                    for (int v = 0; v < NV; v += 2) {
                        const T gx0 = rx * fx[v], gx1 = rx * fx[v + 1], gy0 = ry * fy[v], gy1 = ry * fy[v + 1];
#pragma unroll
                        for (int m = 0; m < NM; ++m) {
                            if (tb.gx[q][m] != 0.0) pfma(vol[v][m], vol[v + 1][m], gx0, gx1, T(tb.gx[q][m]));
                            if (tb.gy[q][m] != 0.0) pfma(vol[v][m], vol[v + 1][m], gy0, gy1, T(tb.gy[q][m]));
                        }
                    }
                } else {
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const T gxv = rx * fx[v], gyv = ry * fy[v];
#pragma unroll
                        for (int m = 0; m < NM; ++m) {
                            if (tb.gx[q][m] != 0.0) vol[v][m] += gxv * T(tb.gx[q][m]);
                            if (tb.gy[q][m] != 0.0) vol[v][m] += gyv * T(tb.gy[q][m]);
                        }
                    }
                }
            };
            // a mirrored pair of points (q at xi, its mirror at -xi): w_q dphi/dxi
            // changes sign with (-1)^(i-1) and w_q dphi/deta with (-1)^i, so
            // each mode takes the sum or the difference of the two points'
            // fluxes: one product per mode and direction for both points
            auto vol_pair = [&](const int q, const T (&uq)[NV], const T (&uqm)[NV]) {
                T fx[NV], fy[NV], hx[NV], hy[NV];
                ph.flux2(uq, fx, fy);
                ph.flux2(uqm, hx, hy);
                if constexpr (NV % 2 == 0) {
#pragma unroll
                    for (int v = 0; v < NV; v += 2) {
                        T sx0, sx1, dx0, dx1, sy0, sy1, dy0, dy1;
                        padd(sx0, sx1, fx[v], fx[v + 1], hx[v], hx[v + 1]);
                        psub(dx0, dx1, fx[v], fx[v + 1], hx[v], hx[v + 1]);
                        padd(sy0, sy1, fy[v], fy[v + 1], hy[v], hy[v + 1]);
                        psub(dy0, dy1, fy[v], fy[v + 1], hy[v], hy[v + 1]);
                        pmul(sx0, sx1, rx);
                        pmul(dx0, dx1, rx);
                        pmul(sy0, sy1, ry);
                        pmul(dy0, dy1, ry);
#pragma unroll
                        for (int m = 0; m < NM; ++m) {
                            if (tb.gx[q][m] != 0.0) {
                                if (tb.ip[m] == 0) pfma(vol[v][m], vol[v + 1][m], dx0, dx1, T(tb.gx[q][m]));
                                else pfma(vol[v][m], vol[v + 1][m], sx0, sx1, T(tb.gx[q][m]));
                            }
                            if (tb.gy[q][m] != 0.0) {
                                if (tb.ip[m] == 0) pfma(vol[v][m], vol[v + 1][m], sy0, sy1, T(tb.gy[q][m]));
                                else pfma(vol[v][m], vol[v + 1][m], dy0, dy1, T(tb.gy[q][m]));
                            }
                        }
                    }
                } else {
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const T sxv = rx * (fx[v] + hx[v]), dxv = rx * (fx[v] - hx[v]);
                        const T syv = ry * (fy[v] + hy[v]), dyv = ry * (fy[v] - hy[v]);
#pragma unroll
                        for (int m = 0; m < NM; ++m) {
                            if (tb.gx[q][m] != 0.0) vol[v][m] += (tb.ip[m] == 0 ? dxv : sxv) * T(tb.gx[q][m]);
                            if (tb.gy[q][m] != 0.0) vol[v][m] += (tb.ip[m] == 0 ? syv : dyv) * T(tb.gy[q][m]);
                        }
                    }
                }
            };
            // point values in mirrored pairs: phi_m(-xi, eta) = (-1)^i phi_m(xi,
            // eta), so the values at xi_a and at -xi_a are the sum and the
            // difference of the even-i and odd-i parts of one contraction (the
            // middle column xi = 0 has no odd part)
#pragma unroll
            for (int q = 0; q < NQV; ++q) {
                const int qa = q / NQ, qb = q % NQ, qm = (NQ - 1 - qa) * NQ + qb;
                if (qa > NQ - 1 - qa) continue;   // evaluated with its mirror point
                T uq[NV], uqm[NV];
                if constexpr (NV % 2 == 0) {
#pragma unroll
                    for (int v = 0; v < NV; v += 2) {
                        T e0 = T(0), e1 = T(0), o0 = T(0), o1 = T(0);
#pragma unroll
                        for (int m = 0; m < NM; ++m)   // (P_1 vanishes at the middle Gauss point)
                            if (tb.phi[q][m] != 0.0) {
                                if (tb.ip[m] == 0) pfma(e0, e1, w[v][m], w[v + 1][m], T(tb.phi[q][m]));
                                else pfma(o0, o1, w[v][m], w[v + 1][m], T(tb.phi[q][m]));
                            }
                        padd(uq[v], uq[v + 1], e0, e1, o0, o1);
                        psub(uqm[v], uqm[v + 1], e0, e1, o0, o1);
                    }
                } else {
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        T e = T(0), o = T(0);
#pragma unroll
                        for (int m = 0; m < NM; ++m)
                            if (tb.phi[q][m] != 0.0) {
                                if (tb.ip[m] == 0) e += w[v][m] * T(tb.phi[q][m]);
                                else o += w[v][m] * T(tb.phi[q][m]);
                            }
                        uq[v] = e + o;
                        uqm[v] = e - o;
                    }
                }
                if (qa < NQ - 1 - qa) vol_pair(q, uq, uqm);
                else vol_point(q, uq);
            }
            if (need_flux && out_row) {
                if constexpr (NV % 2 == 0) {
#pragma unroll
                    for (int v = 0; v < NV; v += 2)
#pragma unroll
                        for (int m = 0; m < NM; ++m) pfma(V[v][m], V[v + 1][m], vol[v][m], vol[v + 1][m], bi);
                } else {
#pragma unroll
                    for (int v = 0; v < NV; ++v)
#pragma unroll
                        for (int m = 0; m < NM; ++m) V[v][m] += bi * vol[v][m];
                }
            }
            // face traces.  phi_m(-1, eta) = (-1)^i phi_m(1, eta): the east and
            // west traces are the sum and difference of the even-i and odd-i
            // parts of one contraction (north and south likewise in j)
            T tE[NQ][NV], tW[NQ][NV], tN[NQ][NV], tS[NQ][NV];
            if constexpr (NV % 2 == 0) {
#pragma unroll
                for (int p = 0; p < NQ; ++p)
#pragma unroll
                    for (int v = 0; v < NV; v += 2) {
                        T xe0 = 0, xe1 = 0, xo0 = 0, xo1 = 0, ye0 = 0, ye1 = 0, yo0 = 0, yo1 = 0;
#pragma unroll
                        for (int m = 0; m < NM; ++m) {
                            if (tb.tE[p][m] != 0.0) {
                                if (tb.ip[m] == 0) pfma(xe0, xe1, w[v][m], w[v + 1][m], T(tb.tE[p][m]));
                                else pfma(xo0, xo1, w[v][m], w[v + 1][m], T(tb.tE[p][m]));
                            }
                            if (tb.tN[p][m] != 0.0) {
                                if (tb.jp[m] == 0) pfma(ye0, ye1, w[v][m], w[v + 1][m], T(tb.tN[p][m]));
                                else pfma(yo0, yo1, w[v][m], w[v + 1][m], T(tb.tN[p][m]));
                            }
                        }
                        padd(tE[p][v], tE[p][v + 1], xe0, xe1, xo0, xo1);
                        psub(tW[p][v], tW[p][v + 1], xe0, xe1, xo0, xo1);
                        padd(tN[p][v], tN[p][v + 1], ye0, ye1, yo0, yo1);
                        psub(tS[p][v], tS[p][v + 1], ye0, ye1, yo0, yo1);
                    }
            } else {
#pragma unroll
            for (int p = 0; p < NQ; ++p)
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    T e = 0, ww = 0, n = 0, s = 0;
#pragma unroll
                    for (int m = 0; m < NM; ++m) {
                        e += w[v][m] * T(tb.tE[p][m]);
                        ww += w[v][m] * T(tb.tW[p][m]);
                        n += w[v][m] * T(tb.tN[p][m]);
                        s += w[v][m] * T(tb.tS[p][m]);
                    }
                    tE[p][v] = e; tW[p][v] = ww; tN[p][v] = n; tS[p][v] = s;
                }
            }
            // local operator L_i = cm (face_loc - vol), eq. (2.7)
            if (need_L) {
                T floc[NV][NM];
#pragma unroll
                for (int v = 0; v < NV; ++v)
#pragma unroll
                    for (int m = 0; m < NM; ++m) floc[v][m] = T(0);
#pragma unroll
                for (int p = 0; p < NQ; ++p) {
                    T fe[NV], fw[NV], fn[NV], fs[NV];
                    ph.template fluxn<0>(tE[p], fe);
                    ph.template fluxn<0>(tW[p], fw);
                    ph.template fluxn<1>(tN[p], fn);
                    ph.template fluxn<1>(tS[p], fs);
                    if constexpr (NV % 2 == 0) {
                        // pW = (-1)^i pE, pS = (-1)^j pN: fe pE - fw pW = pE (fe -+ fw)
#pragma unroll
                        for (int v = 0; v < NV; v += 2) {
                            T xm0, xm1, xp0, xp1, ym0, ym1, yp0, yp1;
                            psub(xm0, xm1, fe[v], fe[v + 1], fw[v], fw[v + 1]);
                            padd(xp0, xp1, fe[v], fe[v + 1], fw[v], fw[v + 1]);
                            psub(ym0, ym1, fn[v], fn[v + 1], fs[v], fs[v + 1]);
                            padd(yp0, yp1, fn[v], fn[v + 1], fs[v], fs[v + 1]);
                            if constexpr (!SQ) {
                                pmul(xm0, xm1, rx);
                                pmul(xp0, xp1, rx);
                                pmul(ym0, ym1, ry);
                                pmul(yp0, yp1, ry);
                            }
#pragma unroll
                            for (int m = 0; m < NM; ++m) {
                                if (tb.pE[p][m] != 0.0) {
                                    if (tb.ip[m] == 0) pfma(floc[v][m], floc[v + 1][m], xm0, xm1, T(tb.pE[p][m]));
                                    else pfma(floc[v][m], floc[v + 1][m], xp0, xp1, T(tb.pE[p][m]));
                                }
                                if (tb.pN[p][m] != 0.0) {
                                    if (tb.jp[m] == 0) pfma(floc[v][m], floc[v + 1][m], ym0, ym1, T(tb.pN[p][m]));
                                    else pfma(floc[v][m], floc[v + 1][m], yp0, yp1, T(tb.pN[p][m]));
                                }
                            }
                        }
                    } else {
#pragma unroll
                        for (int v = 0; v < NV; ++v)
#pragma unroll
                            for (int m = 0; m < NM; ++m)
                                floc[v][m] += rxv * (fe[v] * T(tb.pE[p][m]) - fw[v] * T(tb.pW[p][m])) +
                                              ryv * (fn[v] * T(tb.pN[p][m]) - fs[v] * T(tb.pS[p][m]));
                    }
                }
#pragma unroll
                for (int v = 0; v < NV; ++v)
#pragma unroll
                    for (int m = 0; m < NM; ++m)
                        slot(i * C::NDOF + v * NM + m) =
                            T(tb.cm[m]) * (SQ ? fma(rx, floc[v][m], -vol[v][m]) : floc[v][m] - vol[v][m]);
            }
            if (!need_flux) continue;
            // east face: own east trace vs. the west trace of the lane to the right
            if (out_row) {
                T tWn[NQ][NV], dcE[NV];   // DEV: east neighbour's base minus this cell's
                if constexpr (DEV) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) dcE[v] = shfl_down(cb[v], 1) - cb[v];
                }
#pragma unroll
                for (int p = 0; p < NQ; ++p)
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        tWn[p][v] = shfl_down(tW[p][v], 1);
                        if constexpr (DEV) tWn[p][v] += dcE[v];
                    }
                // boundary strips: the whole warp forms the exterior states (no
                // divergent branch), only the lane at the boundary keeps them
                if (has_bcW) {
                    const bool edge = lane == 0;
                    const BCSide& bcw = a.bc[0];
                    if (bcw.affine) {
#pragma unroll
                        for (int p = 0; p < NQ; ++p)
#pragma unroll
                            for (int v = 0; v < NV; ++v) {
                                T k0 = sizeof(T) == 4 ? T(bcw.cf[v]) : T(bcw.cd[v]);
                                if constexpr (DEV) k0 = fma(T(bcw.m[v]) - T(1), cb[v], k0);
                                const T ext = fma(T(bcw.m[v]), tWn[p][v], k0);
                                tE[p][v] = edge ? ext : tE[p][v];
                            }
                    } else {
                        cold_branch();
                        const int ryc = opaque(ry_), ic = opaque(i);
#pragma unroll
                        for (int p = 0; p < NQ; ++p) {
                            T ext[NV];
                            bcx(bcw, 0, tWn[p], [&](double& x, double& y, double& t) {
                                x = pv.x0();
                                y = pv.y0() + (ryc + 0.5 + 0.5 * tb.xq[p]) * pv.dy();
                                t = t0 + tab_c(a, ic) * dt;
                            }, ext);
#pragma unroll
                            for (int v = 0; v < NV; ++v) tE[p][v] = edge ? ext[v] : tE[p][v];
                        }
                    }
                }
                if (has_bcE) {
                    const bool edge = col == nx - 1;
                    const BCSide& bce = a.bc[1];
                    if (bce.affine) {
#pragma unroll
                        for (int p = 0; p < NQ; ++p)
#pragma unroll
                            for (int v = 0; v < NV; ++v) {
                                T k0 = sizeof(T) == 4 ? T(bce.cf[v]) : T(bce.cd[v]);
                                if constexpr (DEV) k0 = fma(T(bce.m[v]) - T(1), cb[v], k0);
                                const T ext = fma(T(bce.m[v]), tE[p][v], k0);
                                tWn[p][v] = edge ? ext : tWn[p][v];
                            }
                    } else {
                        cold_branch();
                        const int ryc = opaque(ry_), ic = opaque(i);
#pragma unroll
                        for (int p = 0; p < NQ; ++p) {
                            T ext[NV];
                            bcx(bce, 0, tE[p], [&](double& x, double& y, double& t) {
                                x = pv.x0() + nx * pv.dx();
                                y = pv.y0() + (ryc + 0.5 + 0.5 * tb.xq[p]) * pv.dy();
                                t = t0 + tab_c(a, ic) * dt;
                            }, ext);
#pragma unroll
                            for (int v = 0; v < NV; ++v) tWn[p][v] = edge ? ext[v] : tWn[p][v];
                        }
                    }
                }
#pragma unroll
                for (int p = 0; p < NQ; ++p) {
                    T F[NV];
                    llf_ax<0, false>(ph, tE[p], tWn[p], F);
#pragma unroll
                    for (int v = 0; v < NV; ++v) FE[p][v] = fma(hbi, F[v], FE[p][v]);
                }
            }
            // south face: north trace of the row below (stored) vs. own south trace
            if (do_south) {
                T lo[NQ][NV];
                if (south_bc) {   // row 0 without periodic wrap: boundary data (one uniform branch per row)
                    cold_branch();
                    const int colc = opaque(col), ic = opaque(i);
#pragma unroll
                    for (int p = 0; p < NQ; ++p)
                        bcx(a.bc[2], 1, tS[p], [&](double& x, double& y, double& t) {
                            x = pv.x0() + (colc + 0.5) * pv.dx() + 0.5 * pv.dx() * tb.xq[p];
                            y = pv.y0();
                            t = t0 + tab_c(a, ic) * dt;
                        }, lo[p]);
                } else {
#pragma unroll
                    for (int p = 0; p < NQ; ++p)
#pragma unroll
                        for (int v = 0; v < NV; ++v) {
                            lo[p][v] = slot(offN + (i * NQ + p) * NV + v);
                            if constexpr (DEV) lo[p][v] += cS[v] - cb[v];
                        }
                }
#pragma unroll
                for (int p = 0; p < NQ; ++p) {
                    T F[NV];
                    llf_ax<1, false>(ph, lo[p], tS[p], F);
#pragma unroll
                    for (int v = 0; v < NV; ++v) FS[p][v] = fma(hbi, F[v], FS[p][v]);
                }
            }
            // traces for the row above, or for the seams at the segment's ends
            if (keep_north) {
#pragma unroll
                for (int p = 0; p < NQ; ++p)
#pragma unroll
                    for (int v = 0; v < NV; ++v) slot(offN + (i * NQ + p) * NV + v) = tN[p][v];
            } else if (SEAM && outlane) {
#pragma unroll
                for (int p = 0; p < NQ; ++p)
#pragma unroll
                    for (int v = 0; v < NV; ++v) *sc.north(seg, (i * NQ + p) * NV + v, col) = tN[p][v];
            }
            if (SEAM && seam_row && outlane) {
#pragma unroll
                for (int p = 0; p < NQ; ++p)
#pragma unroll
                    for (int v = 0; v < NV; ++v) *sc.south(seg, (i * NQ + p) * NV + v, col) = tS[p][v];
            }
        }

        // ---- finish the row below: its north face is this row's south face --------
        auto finish = [&](T (&P)[NV][NM], int rw) {
            if (!outlane) return;
            store_cell<T, PHYS, NV, NM, COMP>(a, pv, uin, uout, plane, (size_t)rw * nx + col, P, rx, ry, gm1, gam, red);
        };
        // an update that a seam completes, left in the output buffer (COMP: in the hi planes)
        auto leave = [&](const T (&P)[NV][NM], int rw) {
            if (!outlane) return;
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int m = 0; m < NM; ++m) uout[(size_t)(v * NM + m) * plane + (size_t)rw * nx + col] = P[v][m];
        };
        if (do_south && r - 1 >= r0 && r - 1 < r1) {
            // DEV: FS is relative to this row's base; the row below takes it
            // relative to its own: minus f_y(c_below) - f_y(c) (sum_i b_i = 1)
            T gS[NV];
            if constexpr (DEV) {
                T dcS[NV];
#pragma unroll
                for (int v = 0; v < NV; ++v) dcS[v] = cS[v] - cb[v];
                ph.template fluxn<1>(dcS, gS);
            }
            if (SEAM && r - 1 == r0 && seamS) {   // the seam completes the row below: its north flux
                if (outlane) {
#pragma unroll
                    for (int p = 0; p < NQ; ++p)
#pragma unroll
                        for (int v = 0; v < NV; ++v) *sc.flux(seg, p * NV + v, col) = FS[p][v];
                    if constexpr (DEV)
#pragma unroll
                        for (int v = 0; v < NV; ++v) *sc.flux(seg, NQ * NV + v, col) = gS[v];
                }
            } else {
                T P[NV][NM];
#pragma unroll
                for (int v = 0; v < NV; ++v)
#pragma unroll
                    for (int m = 0; m < NM; ++m) P[v][m] = slot(offP + v * NM + m);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    T Fv[NQ];
                    column<NQ, NV>(FS, v, Fv);
                    add_north<T, K, B, DEV>(P[v], Fv, DEV ? gS[v] : T(0), ry, tdt);
                }
                finish(P, r - 1);
            }
        }

        if (!out_row) continue;

        // ---- this row: east/west/south faces and the volume term ----------------------
        // DEV: FE of the lane to the left is relative to its base; moved to this
        // cell's: plus f_x(c_west) - f_x(c)
        T FW[NQ][NV];
#pragma unroll
        for (int p = 0; p < NQ; ++p)
#pragma unroll
            for (int v = 0; v < NV; ++v) FW[p][v] = shfl_up(FE[p][v], 1);
        if constexpr (DEV) {
            T gW[NV], dcW[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) dcW[v] = shfl_up(cb[v], 1) - cb[v];
            ph.template fluxn<0>(dcW, gW);
#pragma unroll
            for (int p = 0; p < NQ; ++p)
#pragma unroll
                for (int v = 0; v < NV; ++v) FW[p][v] += gW[v];
        }
        // east and west faces: pW = (-1)^i pE, so FE pE - FW pW = pE (FE -+ FW)
        T FEm[NQ][NV], FEp[NQ][NV];
#pragma unroll
        for (int p = 0; p < NQ; ++p)
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                FEm[p][v] = FE[p][v] - FW[p][v];
                FEp[p][v] = FE[p][v] + FW[p][v];
            }
        T P[NV][NM];   // first the east/west face terms, then the update
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                T sx = T(0);
#pragma unroll
                for (int p = 0; p < NQ; ++p)
                    if (tb.pE[p][m] != 0.0) sx = fma(tb.ip[m] == 0 ? FEm[p][v] : FEp[p][v], T(tb.pE[p][m]), sx);
                P[v][m] = sx;
            }
        if (SEAM && seam_row) {
            if (outlane)
#pragma unroll
                for (int v = 0; v < NV; ++v)
#pragma unroll
                    for (int m = 0; m < NM; ++m) {
                        *sc.vol(seg, v * NM + m, col) = V[v][m];
                        if (LIM && a.limit) *sc.un(seg, v * NM + m, col) = un[v][m];
                    }
        } else {
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                T Fv[NQ];
                column<NQ, NV>(FS, v, Fv);
                row_update<T, K, B, COMP, SQ>(P[v], P[v], V[v], Fv, un[v], rx, ry, tdt);
            }
        }
        if (r == ny - 1 && !pery) {
            // top boundary: north face flux from the stored north traces
            cold_branch();
            const int colc = opaque(col);
            T FN[NQ][NV];
#pragma unroll
            for (int p = 0; p < NQ; ++p)
#pragma unroll
                for (int v = 0; v < NV; ++v) FN[p][v] = T(0);
            for (int i = 0; i < S; ++i) {
                const T bi = tab_bT<T>(a, i);
                if (bi == T(0)) continue;
                const double ti = t0 + tab_c(a, i) * dt;
#pragma unroll
                for (int p = 0; p < NQ; ++p) {
                    T lo[NV], hi[NV], F[NV];
#pragma unroll
                    for (int v = 0; v < NV; ++v) lo[v] = slot(offN + (i * NQ + p) * NV + v);
                    bcx(a.bc[3], 1, lo, [&](double& x, double& y, double& t) {
                        x = pv.x0() + (colc + 0.5) * pv.dx() + 0.5 * pv.dx() * tb.xq[p];
                        y = pv.y0() + ny * pv.dy();
                        t = ti;
                    }, hi);
                    llf_ax<1>(ph, lo, hi, F);
#pragma unroll
                    for (int v = 0; v < NV; ++v) FN[p][v] = fma(bi, F[v], FN[p][v]);
                }
            }
            if (SEAM && seam_row) {
                if (outlane) {
#pragma unroll
                    for (int p = 0; p < NQ; ++p)
#pragma unroll
                        for (int v = 0; v < NV; ++v) *sc.flux(seg, p * NV + v, col) = FN[p][v];
                    if constexpr (DEV)   // already relative to this row's base
#pragma unroll
                        for (int v = 0; v < NV; ++v) *sc.flux(seg, NQ * NV + v, col) = T(0);
                }
                leave(P, r);
            } else {
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    T Fv[NQ];
                    column<NQ, NV>(FN, v, Fv);
                    add_north<T, K, B, false>(P[v], Fv, T(0), ry, tdt);
                }
                finish(P, r);
            }
        } else if (SEAM && (seam_row || last)) {
            leave(P, r);
        } else {
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int m = 0; m < NM; ++m) slot(offP + v * NM + m) = P[v][m];
        }
    }

    // ---- FP64 reductions: warp -> per-warp slot -> the launch that ends the step -----
    red.template close<PHYS>(outlane && r0 < r1 ? adv_speed : 0.0);
    step_epilogue<NV, C::NRED>(pv, gw, lane, red.max, red.sum, red_trouble, red.status);
}

// One problem: the launch arguments describe the mesh; dt and t come from
// the arguments or from the device run state (device-driven runs).
// (FP64 always leaves its seams to the seam launches: see use_seams)
template <class T, int K, int B, int PHYS, bool COMP = false, bool MLPI = false, bool LIM = true, bool DEV = false,
          bool SQ = false, bool SEAM = sizeof(T) == 8>
__global__ void __launch_bounds__(CRK_STEP_MAXT, PHYS == PHYS_ADV ? CRK_STEP_MINB_ADV : CRK_STEP_MINB2)
    step2d_kernel(const StepArgs a) {
    if constexpr (MLPI) {
        extern __shared__ __align__(16) unsigned char smem_raw[];
        MlpSmem& mw = *reinterpret_cast<MlpSmem*>(smem_raw + mlp_smem_offset<T, K, B, PHYS>(a.s, blockDim.x));
        mlp_load_smem(mw, a.mlp);
        __syncthreads();
    }
    allow_dependent_launch();
    const int gw = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (gw >= a.n_strips * a.n_segs) return;   // whole warp leaves; no block barriers
    const ArgsView<T> pv{a, a.dt_from_dev ? a.ds->t : a.t, a.dt_from_dev ? a.ds->dt : a.dt};
    step2d_body<T, K, B, PHYS, COMP, MLPI, LIM, DEV, SQ, SEAM>(a, pv, gw);
}

template <class T>
constexpr int SEAM_THREADS = sizeof(T) == 4 ? SEAM_THREADS_F32 : SEAM_THREADS_F64;

// The step's second launch: the fluxes sum_i b_i fhat of the seams, one thread
// per (seam, face point, column), columns fastest, all stages' traces loaded
// before they are used.  DEV: relative to the upper row's base; the move to
// the lower row's is stored with it.  (One thread per cell forming the fluxes
// of its own seams and completing the cell did them twice and in fewer threads:
// 0.151 ms against 0.054 + 0.048 for FP64 P^2 on 640 x 160, 0.086 against 0.018 +
// 0.019 for Q^2 RK4 on 80 x 80.)
template <class T, int K, int B, int PHYS, bool DEV, class PV>
__device__ __forceinline__ void seam_flux_body(const StepArgs& a, const PV& pv, int id, bool limited) {
    using C = Step2D<T, K, B, PHYS>;
    constexpr int NQ = C::NQ, NV = C::NV;
    const int nx = pv.nx(), ny = pv.ny(), nseg = pv.n_segs(), S = a.s;
    const int row = id / nx, col = id - row * nx;
    const int s = row / NQ, p = row - s * NQ;   // the seam below segment s
    if (s >= nseg || !(pv.dt() > 0.0)) return;
    if (s == 0 && a.bc[2].type != BC_PERIODIC) return;
    const int sl = s > 0 ? s - 1 : nseg - 1;
    const Seam<T, K, B, PHYS, DEV> sc(pv.seam(), S, nx, limited);
    std::conditional_t<DEV, EulerDev<T>, Phys<T, PHYS>> ph;
    if constexpr (PHYS == PHYS_EULER) {
        ph.gamma = T(a.gamma);
        ph.gm1 = T(a.gamma - 1.0);
    } else {
        ph.bx = T(a.beta[0]);
        ph.by = T(a.beta[1]);
    }
    T lo[MAXS][NV], hi[MAXS][NV], bs[MAXS];
#pragma unroll
    for (int i = 0; i < MAXS; ++i) {
        bs[i] = i < S ? tab_bT<T>(a, i) : T(0);
        if (bs[i] != T(0))
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                lo[i][v] = *sc.north(sl, (i * NQ + p) * NV + v, col);
                hi[i][v] = *sc.south(s, (i * NQ + p) * NV + v, col);
            }
    }
    T dc[NV], gS[NV];
    if constexpr (DEV) {
        const size_t plane = (size_t)nx * ny;
        const int ru = seg_row(s, ny, nseg), rl = ru > 0 ? ru - 1 : ny - 1;
        const T* __restrict__ uin = pv.uin();
        T cu[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            cu[v] = uin[(size_t)(v * C::NM) * plane + (size_t)ru * nx + col];
            dc[v] = uin[(size_t)(v * C::NM) * plane + (size_t)rl * nx + col] - cu[v];
        }
        ph.set_base(cu);
        if (p == 0) {
            ph.template fluxn<1>(dc, gS);
#pragma unroll
            for (int v = 0; v < NV; ++v) *sc.below(s, NQ * NV + v, col) = gS[v];
        }
    }
    T F[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) F[v] = T(0);
#pragma unroll
    for (int i = 0; i < MAXS; ++i) {
        if (bs[i] == T(0)) continue;
        const T hbi = T(0.5) * bs[i];
        if constexpr (DEV)
#pragma unroll
            for (int v = 0; v < NV; ++v) lo[i][v] += dc[v];
        T G[NV];
        llf_ax<1, false>(ph, lo[i], hi[i], G);
#pragma unroll
        for (int v = 0; v < NV; ++v) F[v] = fma(hbi, G[v], F[v]);
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) *sc.below(s, p * NV + v, col) = F[v];
}

template <class T, int K, int B, int PHYS, bool DEV>
__global__ void __launch_bounds__(SEAM_THREADS<T>) seam_flux_kernel(const StepArgs a, bool limited) {
    wait_for_step();
    allow_dependent_launch();
    const ArgsView<T> pv{a, a.dt_from_dev ? a.ds->t : a.t, a.dt_from_dev ? a.ds->dt : a.dt};
    seam_flux_body<T, K, B, PHYS, DEV>(a, pv, blockIdx.x * SEAM_THREADS<T> + threadIdx.x, limited);
}

// The third launch: one thread per variable of a cell of a segment's first or
// last row completes it: a warp per 32 cells (columns fastest) and variable, so
// that a thread holds a quarter of a cell's loads and registers; the averages
// meet in shared memory for the wave speed.  Block blk of nblk takes its share of
// the cells and of the step warps' slots; the last block to arrive (an atomic
// counter, no waiting) reduces the blocks' slots in a fixed order and updates
// the run state.  At most two blocks per SM (seam_blocks): a block per 32 cells
// took longer wherever they were many (FP32 P^2 on 1920 x 480 in segments of 4
// rows, 4 steps: 1.46 against 1.29 ms: FP64 block reductions and the counter).
template <class T, int K, int B, int PHYS, bool COMP, bool DEV, bool SQ, class PV>
__device__ __forceinline__ void seam_body(const StepArgs& a, const PV& pv, int blk, int nblk) {
    using C = Step2D<T, K, B, PHYS>;
    constexpr int NQ = C::NQ, NM = C::NM, NV = C::NV, NT = SEAM_CELL_THREADS, G = NT / (32 * NV);
    __shared__ T avg[G][NV][32];
    const double dt = pv.dt();
    if (!(dt > 0.0)) return;   // the step left the state and the run state unchanged
    const int nx = pv.nx(), ny = pv.ny(), nseg = pv.n_segs();
    const size_t plane = (size_t)nx * ny;
    const bool pery = a.bc[2].type == BC_PERIODIC, limited = !COMP && a.limit;
    const Seam<T, K, B, PHYS, DEV> sc(pv.seam(), a.s, nx, limited);
    const T rx = pv.rxT(), ry = pv.ryT(), tdt = T(dt);
    T gam, gm1;
    if constexpr (sizeof(T) == 4) {
        gam = a.gammaf;
        gm1 = a.gm1f;
    } else {
        gam = a.gamma;
        gm1 = a.gamma - 1.0;
    }
    const T* __restrict__ uin = pv.uin();
    T* __restrict__ uout = pv.uout();
    const int lane = threadIdx.x & 31, v = (threadIdx.x >> 5) % NV, grp = threadIdx.x / (32 * NV);
    const int both = nseg != ny;   // cells by (segment, first or last row, column), or (segment, column)
    const int groups = (int)(((long long)nx * nseg * (1 + both) + 31) / 32);
    T hi = T(0), lo = T(0), fastest = T(0);   // total of this thread's variable, hi + lo
    unsigned st = 0;
    for (int base = blk * G; base < groups; base += nblk * G) {
        const int cell = (base + grp) * 32 + lane;
        const int row = cell / nx, col = cell - row * nx, seg = row >> both;
        bool wrote = false;
        if (seg < nseg) {
            const int r0 = seg_row(seg, ny, nseg), r1 = seg_row(seg + 1, ny, nseg);
            const bool top = both && (row & 1), one = r1 - r0 == 1;
            // the faces the row waits for: below a first row, above a last one
            const bool south = !top && (seg > 0 || pery), north = (top || one) && (seg + 1 < nseg || pery);
            wrote = top ? north && !one : south || north;
            if (wrote) {
                const size_t o = (size_t)(top ? r1 - 1 : r0) * nx + col;
                T P[NM], V[NM], un[NM], FS[NQ], FN[NQ];
                T gS = T(0);
#pragma unroll
                for (int m = 0; m < NM; ++m) P[m] = uout[(size_t)(v * NM + m) * plane + o];
                // the north face: the seam above, or the flux the step formed
                const int su = seg + 1 < nseg ? seg + 1 : 0;
#pragma unroll
                for (int p = 0; p < NQ; ++p)
                    FN[p] = north ? *sc.below(su, p * NV + v, col) : *sc.flux(seg, p * NV + v, col);
                if constexpr (DEV) gS = north ? *sc.below(su, NQ * NV + v, col) : *sc.flux(seg, NQ * NV + v, col);
                if (south) {
#pragma unroll
                    for (int m = 0; m < NM; ++m) {
                        V[m] = *sc.vol(seg, v * NM + m, col);
                        if constexpr (COMP) un[m] = T(0);
                        else un[m] = limited ? *sc.un(seg, v * NM + m, col) : uin[(size_t)(v * NM + m) * plane + o];
                    }
#pragma unroll
                    for (int p = 0; p < NQ; ++p) FS[p] = *sc.below(seg, p * NV + v, col);
                    row_update<T, K, B, COMP, SQ>(P, P, V, FS, un, rx, ry, tdt);
                }
                add_north<T, K, B, DEV>(P, FN, gS, ry, tdt);
                T al = T(0);
#pragma unroll
                for (int m = 0; m < NM; ++m) {
                    const size_t ix = (size_t)(v * NM + m) * plane + o;
                    if constexpr (COMP) {
                        T h, l;
                        store_comp(uin, uout, ix, (size_t)(NV * NM) * plane, P[m], h, l);
                        if (m == 0) {
                            P[0] = h;
                            al = l;
                        }
                    } else {
                        uout[ix] = P[m];
                    }
                }
                avg[grp][v][lane] = P[0];
                const T sum = hi + P[0];   // TwoSum
                const T bv = sum - hi;
                lo += (hi - (sum - bv)) + (P[0] - bv);
                if constexpr (COMP) lo += al;
                hi = sum;
            }
        }
        __syncthreads();
        if (v == 0 && wrote) {
            T A[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) A[i] = avg[grp][i][lane];
            fastest = fmax(fastest, new_speed<T, PHYS, NV>(a, pv, [&](int i) { return A[i]; }, rx, ry, gm1, gam, st));
        }
        __syncthreads();
    }
    DevState* ds = pv.ds();
    st = __reduce_or_sync(0xffffffffu, st);
    if (lane == 0 && st) atomicOr(&ds->status, st);
    StepRed<NV> sr;
    sr.key = speed_key(double(fastest));
    const double total = double(hi) + double(lo);
#pragma unroll
    for (int i = 0; i < NV; ++i) sr.sum[i] = i == v ? total : 0.0;
    // the block's slot: its cells, and its share of the step warps' slots
    const int nw = pv.total_warps();
    for (int w = blk * NT + threadIdx.x; w < nw; w += nblk * NT) sr.add_slot(pv.partials() + (size_t)w * C::NRED);
    sr.template block_reduce<NT>();
    double* const slots = pv.partials() + (size_t)nw * C::NRED;
    unsigned prev = 0;
    if (threadIdx.x == 0) {
        sr.put_slot(slots + (size_t)blk * C::NRED);
        __threadfence();
        prev = atomicAdd(&ds->counter, 1u);
    }
    if (!__syncthreads_or(threadIdx.x == 0 && prev == (unsigned)nblk - 1)) return;
    __threadfence();
    StepRed<NV> tot;
#pragma unroll 4
    for (int b = threadIdx.x; b < nblk; b += NT) tot.add_slot(slots + (size_t)b * C::NRED);
    tot.template block_reduce<NT>();
    if (threadIdx.x == 0) {
        for (int i = 0; i < NV; ++i) tot.sum[i] *= pv.cell();
        finish_run_state(a, ds, __longlong_as_double((long long)tot.key), tot.sum, NV, double(tot.trouble), pv.t(),
                         dt, ds->cfl, ds->t_end, ds->lim_count, pv.cur(), pv.done());
    }
}

template <class T, int K, int B, int PHYS, bool COMP, bool DEV, bool SQ>
__global__ void __launch_bounds__(SEAM_CELL_THREADS) seam_kernel(const StepArgs a) {
    wait_for_step();
    const ArgsView<T> pv{a, a.dt_from_dev ? a.ds->t : a.t, a.dt_from_dev ? a.ds->dt : a.dt};
    seam_body<T, K, B, PHYS, COMP, DEV, SQ>(a, pv, blockIdx.x, gridDim.x);
}

// launches of the seams after a single-problem step launched with b
template <class T, int K, int B, int PHYS, bool COMP = false, bool DEV = false, bool SQ = false>
inline cudaError_t launch_seam(const StepArgs& b, cudaStream_t st) {
    const cudaError_t e = launch_dependent(&seam_flux_kernel<T, K, B, PHYS, DEV>,
                                           seam_flux_blocks(sizeof(T), K + 1, b.nx, b.n_segs), SEAM_THREADS<T>, st, b,
                                           !COMP && b.limit);
    if (e != cudaSuccess) return e;
    return launch_dependent(&seam_kernel<T, K, B, PHYS, COMP, DEV, SQ>, seam_blocks(Step2D<T, K, B, PHYS>::NV, b.nx, b.ny, b.n_segs, 2 * std::max(1, sm_count())), SEAM_CELL_THREADS,
                            st, b);
}

// Batched ensemble: problems of different sizes and domains share the
// scheme, tableau and boundary types; each has its own state slice, run state
// (t, dt from its own FP64 wave-speed reduction, t_end, status) and buffer
// index.  Warps take (problem, warp) tasks from a flattened table; one block per
// problem ends its step.  A problem whose dt is 0 (it reached t_end) costs
// nothing: its warps return at once.
template <class T, int K, int B, int PHYS>
__device__ __forceinline__ ProbView<T> problem_view(const StepArgs& a, const BatchProblem& pb, int p, DevState* states,
                                                    int* curs, unsigned* done, const T* bufA, T* bufB) {
    DevState* ds = states + p;
    const int cur = curs[p];
    ProbView<T> pv;
    T* A = const_cast<T*>(bufA) + pb.offset;
    T* Bb = bufB + pb.offset;
    pv.uin_ = cur ? Bb : A;
    pv.uout_ = cur ? A : Bb;
    pv.nx_ = pb.nx;
    pv.ny_ = pb.ny;
    pv.x0_ = pb.x0;
    pv.y0_ = pb.y0;
    pv.dx_ = pb.dx;
    pv.dy_ = pb.dy;
    pv.rx_ = pb.rx;
    pv.ry_ = pb.ry;
    pv.M_ = a.M;
    pv.bx_ = a.beta[0];
    pv.by_ = a.beta[1];
    pv.t_ = ds->t;
    pv.dt_ = ds->dt;
    pv.n_strips_ = pb.n_strips;
    pv.n_segs_ = pb.n_segs;
    pv.total_warps_ = pb.n_strips * pb.n_segs;
    pv.partials_ = a.partials + (size_t)pb.slot0 * Step2D<T, K, B, PHYS>::NRED;
    pv.seam_ = static_cast<T*>(a.seam) + pb.seam0;
    pv.ds_ = ds;
    pv.cur_ = curs + p;
    pv.done_ = done;
    return pv;
}

// SQ: problems with square cells (pb.sq) take the square-cell form of the
// step (a branch per task, uniform over the warp), the others the general one.
template <class T, int K, int B, int PHYS, bool LIM = true, bool SQ = false, bool SEAM = sizeof(T) == 8>
__global__ void __launch_bounds__(256) batch_step2d_kernel(const StepArgs a, const BatchProblem* __restrict__ probs,
                                                           const int2* __restrict__ tasks, int n_tasks,
                                                           DevState* states, int* curs, unsigned* done,
                                                           const T* bufA, T* bufB) {
    allow_dependent_launch();
    const int gw = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (gw >= n_tasks) return;
    const int2 tk = tasks[gw];
    const BatchProblem pb = probs[tk.x];
    const ProbView<T> pv = problem_view<T, K, B, PHYS>(a, pb, tk.x, states, curs, done, bufA, bufB);
    if constexpr (SQ) {
        if (pb.sq) {
            step2d_body<T, K, B, PHYS, false, false, LIM, false, true, SEAM>(a, pv, tk.y);
            return;
        }
    }
    step2d_body<T, K, B, PHYS, false, false, LIM, false, false, SEAM>(a, pv, tk.y);
}

// The seams of a batched step: blocks of (problem, block) from two tables
template <class T, int K, int B, int PHYS>
__global__ void __launch_bounds__(SEAM_THREADS<T>)
    batch_seam_flux_kernel(const StepArgs a, const BatchProblem* __restrict__ probs, const int2* __restrict__ tasks,
                           DevState* states, int* curs, unsigned* done, const T* bufA, T* bufB, bool limited) {
    const int2 tk = tasks[blockIdx.x];   // the tables are constant
    const BatchProblem pb = probs[tk.x];
    wait_for_step();
    allow_dependent_launch();
    const ProbView<T> pv = problem_view<T, K, B, PHYS>(a, pb, tk.x, states, curs, done, bufA, bufB);
    seam_flux_body<T, K, B, PHYS, false>(a, pv, tk.y * SEAM_THREADS<T> + threadIdx.x, limited);
}

// SQ: problems with square cells (pb.sq) took the square-cell form of the step
template <class T, int K, int B, int PHYS, bool SQ>
__global__ void __launch_bounds__(SEAM_CELL_THREADS)
    batch_seam_kernel(const StepArgs a, const BatchProblem* __restrict__ probs, const int2* __restrict__ tasks,
                      DevState* states, int* curs, unsigned* done, const T* bufA, T* bufB) {
    const int2 tk = tasks[blockIdx.x];
    const BatchProblem pb = probs[tk.x];
    wait_for_step();
    const ProbView<T> pv = problem_view<T, K, B, PHYS>(a, pb, tk.x, states, curs, done, bufA, bufB);
    if constexpr (SQ) {
        if (pb.sq) {
            seam_body<T, K, B, PHYS, false, false, true>(a, pv, tk.y, pb.n_seam_blocks);
            return;
        }
    }
    seam_body<T, K, B, PHYS, false, false, false>(a, pv, tk.y, pb.n_seam_blocks);
}

// The end of a batched step without seams: one block per problem reduces its
// slots and updates its run state and buffer index
constexpr int BATCH_FINALIZE_THREADS = 128;
template <int NV>
__global__ void __launch_bounds__(BATCH_FINALIZE_THREADS)
    batch_finalize_kernel(const StepArgs a, const BatchProblem* __restrict__ probs, DevState* states, int* curs,
                          unsigned* done) {
    const int p = blockIdx.x;
    const long long slot0 = probs[p].slot0;
    const int total = probs[p].n_strips * probs[p].n_segs;
    const double cell = probs[p].dx * probs[p].dy;
    wait_for_step();
    DevState* ds = states + p;
    const double dt = ds->dt;
    if (!(dt > 0.0)) return;   // the problem has reached t_end
    StepRed<NV> red;
#pragma unroll 4
    for (int w = threadIdx.x; w < total; w += BATCH_FINALIZE_THREADS)
        red.add_slot(a.partials + (size_t)(slot0 + w) * (NV + 2));
    red.template block_reduce<BATCH_FINALIZE_THREADS>();
    if (threadIdx.x == 0) {
        for (int v = 0; v < NV; ++v) red.sum[v] *= cell;
        finish_run_state(a, ds, __longlong_as_double((long long)red.key), red.sum, NV, double(red.trouble), ds->t, dt,
                         ds->cfl, ds->t_end, ds->lim_count, curs + p, done);
    }
}

}  // namespace crk
