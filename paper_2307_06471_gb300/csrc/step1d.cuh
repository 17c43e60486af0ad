// Fused cRKDG time step on a 1D mesh (eq. (2.8)).  A warp owns 30 cells plus
// one halo cell on each side, a cell per lane; each lane runs all RK stages of
// its cell with the local operator (eq. (2.7)), exchanges the final-stage face
// traces with its neighbour lane by shuffles and updates its cell.  With n_steps
// > 1 the blocks of one cluster march n_steps steps in one launch: cells stay
// in registers, a warp's first and last cell go to the neighbouring warps'
// halo lanes through (distributed) shared memory, one cluster barrier a step.
//
// Linear advection takes the modal form (step2d_linear.cuh): s - 1 applications
// of the Legendre derivative, the upwind jump on the inflow face, no point
// values -- 35 instead of 190 FP64 operations a cell for P^2.  A step is bound
// by its FP64 operations where warps share an SM's FP64 pipe and by the
// dependent chain otherwise, so a run spreads its warps over up to 8 SMs (a few
// warps do with one SM, and without the cluster's barrier: run1d_blocks).  160
// cells, P^2, SSP-RK3, FP64, 160 steps: 1.33 ms in one block and quadrature form,
// 0.35 ms so.
#pragma once
#include <cooperative_groups.h>

#include "common.cuh"

namespace crk {

// Most warps per block of a run (launch.h: run1d_blocks)
constexpr int RUN1D_WARPS = 4;

// What a lane needs of the mesh
struct Line {
    int nx, col, lane;
    bool per, bcW, bcE;   // periodic; the warp holds the mesh's first / last cell of a non-periodic mesh
};

// u^{n+1} of the lane's cell from u^n of its warp's cells: general flux
template <class T, int K, int PHYS, int NV, int NM, class Slot>
__device__ __forceinline__ void step1d_cell(const StepArgs& a, const Line& ln, const Phys<T, PHYS>& ph, double t0,
                                            double dt, T rx, const Slot& slot, const T (&un)[NV][NM], T (&out)[NV][NM]) {
    constexpr Tab1D<K> tb = make_tab1d<K>();
    constexpr int NQ = K + 1, NDOF = NV * NM;
    const T tdt = opaque(T(dt));
    const int S = a.s;
    T V[NV][NM], FR[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        FR[v] = T(0);
#pragma unroll
        for (int m = 0; m < NM; ++m) V[v][m] = T(0);
    }
    for (int i = 0; i < S; ++i) {
        const T bi = tab_bT<T>(a, i);
        const bool need_L = i < S - 1;
        if (!need_L && bi == T(0)) continue;
        T w[NV][NM];
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int m = 0; m < NM; ++m) w[v][m] = un[v][m];
        for (int j = 0; j < i; ++j) {
            const T ad = tab_aT<T>(a, i, j);
            if (ad == T(0)) continue;
            const T aij = ad * tdt;
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int m = 0; m < NM; ++m) w[v][m] -= aij * slot(j * NDOF + v * NM + m);
        }
        // volume term sum_q w_q f(u_q) P_m'(xi_q) (scaled by 1/dx)
        T vol[NV][NM];
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int m = 0; m < NM; ++m) vol[v][m] = T(0);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            T uq[NV], f[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                T s = T(0);
#pragma unroll
                for (int m = 0; m < NM; ++m) s += w[v][m] * T(tb.phi[q][m]);
                uq[v] = s;
            }
            ph.template fluxn<0>(uq, f);
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int m = 0; m < NM; ++m)
                    if (tb.g[q][m] != 0.0) vol[v][m] += rx * f[v] * T(tb.g[q][m]);
        }
        T tR[NV], tL[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            T r = 0, l = 0;
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                r += w[v][m] * T(tb.tR[m]);
                l += w[v][m] * T(tb.tL[m]);
            }
            tR[v] = r;
            tL[v] = l;
        }
        if (need_L) {
            T fr[NV], fl[NV];
            ph.template fluxn<0>(tR, fr);
            ph.template fluxn<0>(tL, fl);
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int m = 0; m < NM; ++m)
                    slot(i * NDOF + v * NM + m) =
                        T(tb.cm[m]) * (rx * (fr[v] * T(tb.tR[m]) - fl[v] * T(tb.tL[m])) - vol[v][m]);
        }
        if (bi == T(0)) continue;
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int m = 0; m < NM; ++m) V[v][m] += bi * vol[v][m];
        T tLn[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) tLn[v] = shfl_down(tL[v], 1);
        if (ln.bcW && ln.lane == 0) {
            cold_branch();
            const int ic = opaque(i);
            bc_exterior<T, NV>(a.bc[0], 0, tLn, [&](double& x, double& y, double& t) {
                x = a.x0;
                y = 0.0;
                t = t0 + tab_c(a, ic) * dt;
            }, tR);
        }
        if (ln.bcE && ln.col == ln.nx - 1) {
            cold_branch();
            const int ic = opaque(i);
            bc_exterior<T, NV>(a.bc[1], 0, tR, [&](double& x, double& y, double& t) {
                x = a.x0 + ln.nx * a.dx;
                y = 0.0;
                t = t0 + tab_c(a, ic) * dt;
            }, tLn);
        }
        T F[NV];
        llf<T, PHYS, 0>(ph, tR, tLn, F);
#pragma unroll
        for (int v = 0; v < NV; ++v) FR[v] += bi * F[v];
    }
    T FL[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) FL[v] = shfl_up(FR[v], 1);
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const T face = FR[v] * T(tb.tR[m]) - FL[v] * T(tb.tL[m]);
            out[v][m] = un[v][m] - tdt * T(tb.cm[m]) * (rx * face - V[v][m]);
        }
}

// ... and for the linear flux in modal form
template <class T, int K, int NM>
__device__ __forceinline__ void step1d_linear(const StepArgs& a, const Line& ln, double t0, double dt,
                                              const T (&un)[NM], T (&out)[NM]) {
    constexpr bool F32 = sizeof(T) == 4;
    const T tdt = T(dt), cx = F32 ? T(a.lin_kf[0]) : T(a.lin_k[0]);
    const int S = a.s;
    // D w = (2 b / dx) dw/dxi
    auto applyD = [&](const T (&w)[NM], T (&d)[NM]) {
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            T acc = T(0);
#pragma unroll
            for (int c = m + 1; c < NM; c += 2) acc += w[c];
            d[m] = (cx * T(2 * m + 1)) * acc;
        }
    };
    // sum_i b_i u^(i) = sum_l gamma_l (-dt D)^l u^n
    T w[NM], d[NM];
    bool started = false;
#pragma unroll
    for (int l = MAXS - 1; l >= 0; --l) {
        if (l < S) {
            const T gl = F32 ? T(a.lin_gammaf[l]) : T(a.lin_gamma[l]);
            if (started) {
                applyD(w, d);
#pragma unroll
                for (int m = 0; m < NM; ++m) w[m] = fma(-tdt, d[m], gl * un[m]);
            } else {
#pragma unroll
                for (int m = 0; m < NM; ++m) w[m] = gl * un[m];
                started = true;
            }
        }
    }
    applyD(w, d);
    T tR = T(0), tL = T(0);
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        tR += w[m];
        tL += m % 2 ? -w[m] : w[m];
    }
    T west = shfl_up(tR, 1), east = shfl_down(tL, 1);
    // exterior trace at a boundary on the inflow side, sum_i b_i of the stages'
    // (in: that sum of the interior traces)
    auto exterior = [&](const BCSide& bc, T in, double xb) {
        if (bc.type == BC_OUTFLOW) return in;
        T e = T(0);
        for (int i = 0; i < S; ++i) {
            const T bi = tab_bT<T>(a, i);
            if (bi == T(0)) continue;
            T g;
            bc_exterior<T, 1>(bc, 0, &in, [&](double& x, double& y, double& t) {
                x = xb;
                y = 0.0;
                t = t0 + tab_c(a, i) * dt;
            }, &g);
            e = fma(bi, g, e);
        }
        return e;
    };
    const bool inW = a.lin_inflow & 1, inE = a.lin_inflow & 2;
    if (inW && ln.bcW && ln.col == 0) west = exterior(a.bc[0], tL, a.x0);
    if (inE && ln.bcE && ln.col == ln.nx - 1) east = exterior(a.bc[1], tR, a.x0 + ln.nx * a.dx);
    const T kW = F32 ? T(a.lin_kf[2]) : T(a.lin_k[2]), kE = F32 ? T(a.lin_kf[3]) : T(a.lin_k[3]);
    const T jump = inW ? kW * (west - tL) : (inE ? kE * (east - tR) : T(0));
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        const T s = inW && m % 2 ? T(-(2 * m + 1)) : T(2 * m + 1);
        out[m] = fma(-tdt, fma(s, jump, d[m]), un[m]);
    }
}

// ONE: a single step, or a run of one block, whose warps meet at the block's
// barrier; otherwise a run of one cluster
template <class T, int K, int PHYS, bool ONE>
__global__ void __launch_bounds__(256) step1d_kernel(const StepArgs a, int n_steps) {
    constexpr int NM = K + 1, NV = Phys<T, PHYS>::NV, NDOF = NV * NM;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    __shared__ T halo[2][RUN1D_WARPS][2][NDOF];   // by step parity, warp, west / east
    const int nthr = blockDim.x, tid = threadIdx.x, lane = tid & 31, wpb = nthr >> 5;
    auto slot = [&](int k) -> T& { return sm[k * nthr + tid]; };

    const int nx = a.nx;
    const int gw = blockIdx.x * wpb + (tid >> 5);
    const int xs = gw * 30, n_out = min(30, nx - xs);   // first cell, cells (<= 0: a warp past the mesh)
    Line ln;
    ln.nx = nx;
    ln.lane = lane;
    ln.col = xs - 1 + lane;
    ln.per = a.bc[0].type == BC_PERIODIC;
    ln.bcW = !ln.per && xs == 0;
    ln.bcE = !ln.per && xs + 30 >= nx;
    const int col = ln.col;
    int xl = ((col % nx) + nx) % nx;
    if (!ln.per) xl = col < 0 ? 0 : (col >= nx ? nx - 1 : col);
    const bool outlane = lane >= 1 && lane <= n_out;

    Phys<T, PHYS> ph;
    if constexpr (PHYS == PHYS_ADV) {
        ph.bx = T(a.beta[0]);
        ph.by = T(0);
    } else {
        // (held in registers: formed again at every use they are FP64 arithmetic)
        ph.gamma = opaque(T(a.gamma));
        ph.gm1 = opaque(T(a.gamma - 1.0));
    }
    const T rx = sizeof(T) == 4 ? T(a.rxf) : T(a.rx);
    const T* src = static_cast<const T*>(a.uin);
    const auto cluster = cooperative_groups::this_cluster();
    // a block's shared memory may be written once the block has started: every
    // block says so here, and the first push waits for all of them
    if constexpr (!ONE) cluster.barrier_arrive();
    T un[NV][NM], out[NV][NM];
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int m = 0; m < NM; ++m) un[v][m] = src[(size_t)(v * NM + m) * nx + xl];

    const int warps = (nx + 29) / 30;
    const int gl = gw > 0 ? gw - 1 : warps - 1, gr = gw + 1 < warps ? gw + 1 : 0;   // neighbouring warps
    double t0 = a.t;   // accumulated as a caller that steps accumulates it
    for (int step = 0; step < n_steps; ++step, t0 += a.dt) {
        if (n_out > 0) {
            if constexpr (PHYS == PHYS_ADV) step1d_linear<T, K, NM>(a, ln, t0, a.dt, un[0], out[0]);
            else step1d_cell<T, K, PHYS, NV, NM>(a, ln, ph, t0, a.dt, rx, slot, un, out);
        }
        if (step + 1 == n_steps) break;
        if constexpr (!ONE)
            if (step == 0) cluster.barrier_wait();
        auto push = [&](int warp, int side) {   // to a warp's halo lane
            T* h;
            if constexpr (ONE) h = &halo[step & 1][warp][side][0];
            else h = cluster.map_shared_rank(&halo[step & 1][warp % wpb][side][0], warp / wpb);
#pragma unroll
            for (int v = 0; v < NV; ++v)
#pragma unroll
                for (int m = 0; m < NM; ++m) h[v * NM + m] = out[v][m];
        };
        if (lane == 1 && n_out > 0 && (ln.per || gw > 0)) push(gl, 1);
        if (lane == n_out && n_out > 0 && (ln.per || gw + 1 < warps)) push(gr, 0);
        if constexpr (ONE) __syncthreads();
        else cluster.sync();
        const bool hw = lane == 0 && !ln.bcW, he = lane == n_out + 1 && !ln.bcE;
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                if (outlane) un[v][m] = out[v][m];
                if (hw || he) un[v][m] = halo[step & 1][tid >> 5][he][v * NM + m];
            }
    }
    // the result goes where an odd or even number of ping-pong steps ends (in
    // place only after a barrier: every warp has read its halo cells)
    T* dst = n_steps % 2 ? static_cast<T*>(a.uout) : const_cast<T*>(src);
    if (outlane)
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int m = 0; m < NM; ++m) dst[(size_t)(v * NM + m) * nx + col] = out[v][m];
    // (no block leaves while another may still write to its shared memory: the
    // last barrier follows the last push)
}

}  // namespace crk
