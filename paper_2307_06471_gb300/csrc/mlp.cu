// Learned troubled-cell indicator (no counterpart in the paper): training
// kernels (FP32 forward/backward with a deterministic gradient reduction,
// Adam), BF16 tensor-core inference, and the feature/label extraction from a
// solver state.  C ABI part of include/crkdg.h.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/crkdg.h"
#include "aux_kernels.cuh"
#include "launch.h"
#include "mlp_warp.cuh"
#include "mlp_tc.cuh"

using crk::MLP_H;
using crk::MLP_IN;
using crk::MLP_NPARAM;
using crk::StepArgs;

namespace {

thread_local std::string g_merr;
int mfail(int code, const std::string& m) {
    g_merr = m;
    return code;
}
#define MCK(call)                                                                                    \
    do {                                                                                             \
        cudaError_t e_ = (call);                                                                     \
        if (e_ != cudaSuccess) return mfail(CRKDG_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

// Training: samples per tile of a block, and the strides of the weights' and
// activations' rows in shared memory (multiples of 4 floats that put 8
// consecutive rows in distinct banks: a row each for 8 lanes' 16-byte loads)
constexpr int TILE = 8;
constexpr int SX = 44, SH = 68;
constexpr int TRAIN_THREADS = 256;

// offsets of the packed parameter vector
constexpr int OW1 = 0, OB1 = OW1 + MLP_H * MLP_IN, OW2 = OB1 + MLP_H, OB2 = OW2 + MLP_H * MLP_H,
              OW3 = OB2 + MLP_H, OB3 = OW3 + MLP_H * MLP_H, OW4 = OB3 + MLP_H, OB4 = OW4 + MLP_H;

// The two launches of a minibatch and the next one's follow one another as
// programmatic dependents: a launch's blocks are set up (and the first tile's
// samples read) while the one before runs, and wait here for its completion
// (an epoch of 8000 samples in minibatches of 1024: 0.255 -> 0.243 ms).
__device__ __forceinline__ void wait_for_launch() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_next_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

struct TrainSmem {
    float W1[MLP_H * SX], W2[MLP_H * SH], W3[MLP_H * SH];
    float b1[MLP_H], b2[MLP_H], b3[MLP_H], W4[MLP_H], b4[4];
    float X[TILE * SX], H1[TILE * SH], H2[TILE * SH], H3[TILE * SH];
    float G[TILE * SH], G2[TILE * SH];   // the delta of a layer, and of the one below
    float dz[TILE];
};

// Forward and backward of the mean class-weighted BCE over n samples (rows
// idx[i] of X, labels y; idx null: the rows in order); writes this block's
// gradient contribution (already divided by n) and loss sum.
//
// A minibatch of 1024 samples is small for the GPU, so a tile is 8 samples
// (128 blocks; one wave of larger n walks its tiles) and the block's gradient
// stays in registers (52 values a thread) until its last tile.  Two samples of a
// thread's unit share its weights' 16-byte loads in the forward pass.
// With tiles of 64 samples, a block per tile and unpadded rows (32-way bank
// conflicts on the weights) a minibatch of 1024 took 0.126 ms; this takes
// 0.014 ms (0.023 while the loads of the weights waited for one another).
// What the launch before wrote (the weights) or still reads (gpart, lpart) is
// touched after wait_for_launch only, the weights by loads that are not moved
// before it (__ldcg; __ldg may be).
__global__ void __launch_bounds__(TRAIN_THREADS) mlp_fwdbwd_kernel(const float* __restrict__ prm,
                                                                   const float* __restrict__ X,
                                                                   const float* __restrict__ y,
                                                                   const int* __restrict__ idx, int n, float pos_weight,
                                                                   float* __restrict__ gpart,
                                                                   float* __restrict__ lpart) {
    extern __shared__ __align__(16) unsigned char sh_raw[];
    TrainSmem& sh = *reinterpret_cast<TrainSmem*>(sh_raw);
    const int tid = threadIdx.x, unit = tid & 63, sg = tid >> 6;   // unit of a layer, pair of samples
    allow_next_launch();
    auto load_tile = [&](long long s0) {
        for (int i = tid; i < TILE * MLP_IN; i += TRAIN_THREADS) {
            const int t = i / MLP_IN, k = i % MLP_IN;
            const bool in = s0 + t < n;
            const long long row = in ? (idx ? idx[s0 + t] : s0 + t) : 0;
            sh.X[t * SX + k] = in ? X[(size_t)row * MLP_IN + k] : 0.f;
        }
    };
    const long long first = (long long)blockIdx.x * TILE;
    load_tile(first);
    wait_for_launch();
    // (unrolled: the loads of a matrix are in flight together)
    static_assert(MLP_H * MLP_IN % TRAIN_THREADS == 0 && MLP_H * MLP_H % TRAIN_THREADS == 0, "whole rounds");
#pragma unroll
    for (int r = 0; r < MLP_H * MLP_IN / TRAIN_THREADS; ++r) {
        const int i = r * TRAIN_THREADS + tid;
        sh.W1[i / MLP_IN * SX + i % MLP_IN] = __ldcg(prm + OW1 + i);
    }
#pragma unroll
    for (int r = 0; r < MLP_H * MLP_H / TRAIN_THREADS; ++r) {
        const int i = r * TRAIN_THREADS + tid;
        sh.W2[(i >> 6) * SH + (i & 63)] = __ldcg(prm + OW2 + i);
        sh.W3[(i >> 6) * SH + (i & 63)] = __ldcg(prm + OW3 + i);
    }
    if (tid < MLP_H) {
        sh.b1[tid] = __ldcg(prm + OB1 + tid);
        sh.b2[tid] = __ldcg(prm + OB2 + tid);
        sh.b3[tid] = __ldcg(prm + OB3 + tid);
        sh.W4[tid] = __ldcg(prm + OW4 + tid);
    }
    if (tid == 0) sh.b4[0] = __ldcg(prm + OB4);
    // gradient of this thread's weights: rows sg + 4 i, column `unit`
    float g1[16], g2[16], g3[16], gb1 = 0.f, gb2 = 0.f, gb3 = 0.f, g4 = 0.f, lsum = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) g1[i] = g2[i] = g3[i] = 0.f;

    // out = relu(W in + b) of two samples
    auto dense = [&](const float* in, int nin, int sin, const float* W, const float* b, float* out) {
        const float* w = W + unit * sin;
        const float* x0 = in + 2 * sg * sin;
        float a0 = b[unit], a1 = a0;
#pragma unroll
        for (int k = 0; k < nin; k += 4) {
            const float4 wv = *reinterpret_cast<const float4*>(w + k);
            const float4 u = *reinterpret_cast<const float4*>(x0 + k);
            const float4 v = *reinterpret_cast<const float4*>(x0 + sin + k);
            a0 = fmaf(u.x, wv.x, a0);
            a1 = fmaf(v.x, wv.x, a1);
            a0 = fmaf(u.y, wv.y, a0);
            a1 = fmaf(v.y, wv.y, a1);
            a0 = fmaf(u.z, wv.z, a0);
            a1 = fmaf(v.z, wv.z, a1);
            a0 = fmaf(u.w, wv.w, a0);
            a1 = fmaf(v.w, wv.w, a1);
        }
        out[2 * sg * SH + unit] = fmaxf(a0, 0.f);
        out[(2 * sg + 1) * SH + unit] = fmaxf(a1, 0.f);
        __syncthreads();
    };
    // a layer's gradient (G its delta, `in` its input) added to gw and gb, and
    // the delta below it, gout = (W^T G) where hin > 0
    auto back = [&](const float* G, const float* in, int nin, int sin, const float* W, float* gw, float& gb, float* gout) {
        if (unit < nin) {
            float x[TILE];
#pragma unroll
            for (int t = 0; t < TILE; ++t) x[t] = in[t * sin + unit];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float* g = G + sg + 4 * i;
                float a = gw[i];
#pragma unroll
                for (int t = 0; t < TILE; ++t) a = fmaf(g[t * SH], x[t], a);
                gw[i] = a;
            }
        }
        if (tid < MLP_H)
#pragma unroll
            for (int t = 0; t < TILE; ++t) gb += G[t * SH + tid];
        if (gout) {
            const float* g0 = G + 2 * sg * SH;
            float a0 = 0.f, a1 = 0.f;
#pragma unroll 8
            for (int j = 0; j < MLP_H; ++j) {
                const float w = W[j * SH + unit];
                a0 = fmaf(g0[j], w, a0);
                a1 = fmaf(g0[SH + j], w, a1);
            }
            gout[2 * sg * SH + unit] = in[2 * sg * sin + unit] > 0.f ? a0 : 0.f;
            gout[(2 * sg + 1) * SH + unit] = in[(2 * sg + 1) * sin + unit] > 0.f ? a1 : 0.f;
        }
        __syncthreads();
    };
    for (long long s0 = first; s0 < n; s0 += (long long)gridDim.x * TILE) {
        const int ns = (int)min((long long)TILE, n - s0);
        if (s0 != first) {
            __syncthreads();
            load_tile(s0);
        }
        __syncthreads();
        dense(sh.X, MLP_IN, SX, sh.W1, sh.b1, sh.H1);
        dense(sh.H1, MLP_H, SH, sh.W2, sh.b2, sh.H2);
        dense(sh.H2, MLP_H, SH, sh.W3, sh.b3, sh.H3);
        if (tid < TILE) {
            float z = sh.b4[0];
#pragma unroll 16
            for (int k = 0; k < MLP_H; ++k) z = fmaf(sh.H3[tid * SH + k], sh.W4[k], z);
            float d = 0.f;
            if (tid < ns) {
                const float yy = y[idx ? idx[s0 + tid] : s0 + tid];
                const float ls = -log1pf(expf(-fabsf(z))) + fminf(z, 0.f);       // log sigma(z)
                const float l1s = -log1pf(expf(-fabsf(z))) + fminf(-z, 0.f);     // log(1 - sigma(z))
                lsum += -(pos_weight * yy * ls + (1.f - yy) * l1s);
                const float sgm = 1.f / (1.f + expf(-z));
                d = (pos_weight * yy * (sgm - 1.f) + (1.f - yy) * sgm) / float(n);
            }
            sh.dz[tid] = d;
        }
        __syncthreads();
        // output layer
        if (tid < MLP_H) {
#pragma unroll
            for (int t = 0; t < TILE; ++t) g4 = fmaf(sh.dz[t], sh.H3[t * SH + tid], g4);
        } else if (tid == MLP_H) {
#pragma unroll
            for (int t = 0; t < TILE; ++t) g4 += sh.dz[t];   // the bias
        }
#pragma unroll
        for (int t = 2 * sg; t < 2 * sg + 2; ++t)
            sh.G[t * SH + unit] = sh.H3[t * SH + unit] > 0.f ? sh.dz[t] * sh.W4[unit] : 0.f;
        __syncthreads();
        back(sh.G, sh.H2, MLP_H, SH, sh.W3, g3, gb3, sh.G2);
        back(sh.G2, sh.H1, MLP_H, SH, sh.W2, g2, gb2, sh.G);
        back(sh.G, sh.X, MLP_IN, SX, sh.W1, g1, gb1, nullptr);
    }
    float* gb = gpart + (size_t)blockIdx.x * MLP_NPARAM;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int j = sg + 4 * i;
        if (unit < MLP_IN) gb[OW1 + j * MLP_IN + unit] = g1[i];
        gb[OW2 + j * MLP_H + unit] = g2[i];
        gb[OW3 + j * MLP_H + unit] = g3[i];
    }
    if (tid < MLP_H) {
        gb[OB1 + tid] = gb1;
        gb[OB2 + tid] = gb2;
        gb[OB3 + tid] = gb3;
    }
    if (tid <= MLP_H) gb[OW4 + tid] = g4;   // OB4 follows W4
    // loss partial
    for (int off = 16; off > 0; off >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
    if (tid == 0) lpart[blockIdx.x] = lsum;   // the losses are in the first warp's lanes
}

// Adam (Kingma and Ba): moments and bias-corrected step; prm null: none
struct AdamArgs {
    float *prm, *m, *v;
    float lr, b1, b2, eps, c1, c2;
};

// grad[p] = sum over blocks, four runs of blocks in block order, then their
// sum (deterministic), the loss likewise, and the Adam step of the parameter
constexpr int REDUCE_RUNS = 4, REDUCE_PARAMS = 64;
__global__ void __launch_bounds__(REDUCE_RUNS * REDUCE_PARAMS)
    mlp_reduce_kernel(const float* __restrict__ gpart, const float* __restrict__ lpart, int nblocks, int n,
                      float* __restrict__ grad, double* __restrict__ loss, const AdamArgs ad) {
    __shared__ float part[REDUCE_RUNS][REDUCE_PARAMS];
    const int t = threadIdx.x % REDUCE_PARAMS, run = threadIdx.x / REDUCE_PARAMS;
    const int p = blockIdx.x * REDUCE_PARAMS + t;
    const int per = (nblocks + REDUCE_RUNS - 1) / REDUCE_RUNS;
    allow_next_launch();
    wait_for_launch();
    const int b0 = run * per, b1 = min(nblocks, b0 + per);
    float a = 0.f;
    if (p < MLP_NPARAM)
#pragma unroll 16
        for (int b = b0; b < b1; ++b) a += __ldcg(gpart + (size_t)b * MLP_NPARAM + p);
    part[run][t] = a;
    __syncthreads();
    if (run == 0 && p < MLP_NPARAM) {
        float g = part[0][t];
#pragma unroll
        for (int i = 1; i < REDUCE_RUNS; ++i) g += part[i][t];
        grad[p] = g;
        if (ad.prm) {
            const float mi = ad.b1 * ad.m[p] + (1.f - ad.b1) * g;
            const float vi = ad.b2 * ad.v[p] + (1.f - ad.b2) * g * g;
            ad.m[p] = mi;
            ad.v[p] = vi;
            ad.prm[p] -= ad.lr * (mi / ad.c1) / (sqrtf(vi / ad.c2) + ad.eps);
        }
    }
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        double l = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += 32) l += double(__ldcg(lpart + b));
        for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        if (threadIdx.x == 0) *loss = l / n;
    }
}

// a launch, `dependent`: as the programmatic dependent of the stream's last one
template <class... A, class... V>
cudaError_t launch(void (*kern)(A...), int grid, int threads, size_t smem, bool dependent, cudaStream_t st, V... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, A(args)...);
}

// BF16 tensor-core inference, a warp per 32 samples.  A grid of resident blocks
// loads the weights once per block and walks the samples; the warp reads its
// samples' features as one run of memory and rounds them into its staging area
// (VEC: pairs, where X allows 8-byte loads).  A block per 128 samples that
// loaded the weights each time, lanes reading 160 bytes apart and the weights'
// rows in one bank group took 0.202 ms for 524,288 samples; this takes 0.043 ms.
constexpr int PREDICT_THREADS = 128;
template <bool VEC>
__global__ void __launch_bounds__(PREDICT_THREADS) mlp_predict_kernel(const float* __restrict__ prm,
                                                                      const float* __restrict__ X, int n,
                                                                      float* __restrict__ logits) {
    extern __shared__ __align__(16) unsigned char smb[];
    crk::MlpSmem& w = *reinterpret_cast<crk::MlpSmem*>(smb);
    const int lane = threadIdx.x & 31;
    __nv_bfloat16* stage = reinterpret_cast<__nv_bfloat16*>(smb + sizeof(crk::MlpSmem)) +
                           (threadIdx.x >> 5) * (32 * crk::MLP_INP + 64);
    crk::mlp_load_smem(w, prm);
    // the padding columns 40 .. 47 stay zero
    for (int k = MLP_IN; k < crk::MLP_INP; k += 2) *reinterpret_cast<uint32_t*>(stage + lane * crk::MLP_INP + k) = 0u;
    __syncthreads();
    const long long warps = (long long)gridDim.x * (PREDICT_THREADS / 32);
    for (long long t = (long long)blockIdx.x * (PREDICT_THREADS / 32) + (threadIdx.x >> 5); t * 32 < n; t += warps) {
        const int s0 = (int)(t * 32), ns = min(32, n - s0);
        const float* x = X + (size_t)s0 * MLP_IN;
        constexpr int PAIRS = MLP_IN / 2;
        float2 f[PAIRS];
#pragma unroll
        for (int j = 0; j < PAIRS; ++j) {   // 32 x 20 pairs, pair i of the run
            const int i = j * 32 + lane;
            f[j] = make_float2(0.f, 0.f);
            if (i < ns * PAIRS) {
                if constexpr (VEC) f[j] = __ldg(reinterpret_cast<const float2*>(x) + i);
                else f[j] = make_float2(__ldg(x + 2 * i), __ldg(x + 2 * i + 1));
            }
        }
#pragma unroll
        for (int j = 0; j < PAIRS; ++j) {
            const int i = j * 32 + lane, r = i / PAIRS, k = 2 * (i % PAIRS);
            *reinterpret_cast<uint32_t*>(stage + r * crk::MLP_INP + k) = crk::pack_bf16(f[j].x, f[j].y);
        }
        const float z = crk::mlp_warp_staged2(w, stage);
        if (lane < ns) logits[s0 + lane] = z;
    }
}

// The same inference on the fifth-generation tensor cores (mlp_tc.cuh): one
// tile of 128 samples per block iteration, grid-stride over the tiles; a
// bounded wait that ran out sets ST_TIMEOUT in *status.
__global__ void __launch_bounds__(crk::MLPTC_CELLS) mlp_predict_tc_kernel(const float* __restrict__ prm,
                                                             const float* __restrict__ X, int n,
                                                             float* __restrict__ logits, unsigned* status) {
    extern __shared__ __align__(1024) unsigned char smt[];
    crk::MlpTcSmem& s = *reinterpret_cast<crk::MlpTcSmem*>(smt);
    crk::mlp_tc_setup(s, prm);
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; ok && (long long)tile * crk::MLPTC_CELLS < n; tile += gridDim.x) {
        const int i = tile * crk::MLPTC_CELLS + threadIdx.x;
        float f[MLP_IN];
        for (int k = 0; k < MLP_IN; ++k) f[k] = i < n ? X[(size_t)i * MLP_IN + k] : 0.f;
        float z;
        ok = crk::mlp_tc_logit(s, f, phase, z);
        if (i < n) logits[i] = z;
    }
    if (!ok && threadIdx.x == 0) atomicOr(status, crk::ST_TIMEOUT);
    crk::mlp_tc_teardown(s);
}

// Features and TVB labels of every cell of a P^2 2D Euler state (one thread
// per cell, 128 cells of a row per block).  Label 1 when the TVB-minmod test of
// the limiter flags the cell.  The block's 128 x 40 features leave through
// shared memory as one run (a thread writing its own 160 bytes touched 32
// sectors per store), and the test's constants come from the host (set_derived)
// instead of FP64 products in every thread: 0.106 -> 0.026 ms for 1024 x 512
// FP32 cells.
constexpr int FEAT_THREADS = 128;
template <class T, int K, int B>
__global__ void __launch_bounds__(FEAT_THREADS) features_kernel(const StepArgs a, const T* __restrict__ u,
                                                                float* __restrict__ X, float* __restrict__ y) {
    constexpr int NM = crk::Tab2D<K, B>::NM;
    __shared__ float out[FEAT_THREADS * (MLP_IN + 1)];
    const int nx = a.nx, ny = a.ny;
    const size_t plane = (size_t)nx * ny;
    const int x0 = blockIdx.x * FEAT_THREADS, x = x0 + threadIdx.x;
    const int yy = blockIdx.y;
    if (x < nx) {
        const bool perx = a.bc[0].type == crk::BC_PERIODIC, pery = a.bc[2].type == crk::BC_PERIODIC;
        // every load at a valid (wrapped or clamped) address, ghosts afterwards
        const int ys = yy > 0 ? yy - 1 : (pery ? ny - 1 : 0), yn = yy < ny - 1 ? yy + 1 : (pery ? 0 : ny - 1);
        const int xw = x > 0 ? x - 1 : (perx ? nx - 1 : 0), xe = x < nx - 1 ? x + 1 : (perx ? 0 : nx - 1);
        T c[4][NM], own[4], nbW[4], nbE[4], nbS[4], nbN[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
#pragma unroll
            for (int m = 0; m < NM; ++m) c[v][m] = u[(size_t)(v * NM + m) * plane + (size_t)yy * nx + x];
            const T* p = u + (size_t)(v * NM) * plane;
            nbW[v] = p[(size_t)yy * nx + xw];
            nbE[v] = p[(size_t)yy * nx + xe];
            nbS[v] = p[(size_t)ys * nx + x];
            nbN[v] = p[(size_t)yn * nx + x];
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) own[v] = c[v][0];
        const crk::LimMesh g = crk::single_mesh<T>(a);
        crk::limit2d_ghosts<T, 4>(a, g, x, yy, own, nbW, nbE, nbS, nbN);
        float f[MLP_IN];
        crk::mlp_features<T, NM>(c, nbE, nbW, nbN, nbS, a.mlp_scale, f);
#pragma unroll
        for (int k = 0; k < MLP_IN; ++k) out[threadIdx.x * (MLP_IN + 1) + k] = f[k];
        T gam;
        if constexpr (sizeof(T) == 4) gam = a.gammaf;
        else gam = a.gamma;
        const bool fl = crk::tvb_limit_cell<T, 4, NM>(c, nbW, nbE, nbS, nbN, T(g.Mdx2), T(g.Mdy2), gam);
        y[(size_t)yy * nx + x] = fl ? 1.f : 0.f;
    }
    __syncthreads();
    const int cells = min(FEAT_THREADS, nx - x0);
    float* Xb = X + ((size_t)yy * nx + x0) * MLP_IN;
    for (int i = threadIdx.x; i < cells * MLP_IN; i += FEAT_THREADS) Xb[i] = out[i / MLP_IN * (MLP_IN + 1) + i % MLP_IN];
}

uint64_t splitmix(uint64_t& s) {
    s += 0x9E3779B97F4A7C15ull;
    uint64_t z = s;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
// device memory for at least n values
template <class V>
bool grow(V*& p, size_t& cap, size_t n) {
    if (n <= cap) return true;
    if (p) cudaFree(p);
    p = nullptr;
    cap = 0;
    if (cudaMalloc(&p, n * sizeof(V)) != cudaSuccess) {
        cudaGetLastError();
        p = nullptr;
        return false;
    }
    cap = n;
    return true;
}

// A host buffer that a copy on a stream may still be reading: the copy is done
// once wait() has returned, and before the guard goes.  (Copies from pageable
// memory may return before they have read it where the GPU reads pageable
// memory itself, as it does beside a Grace host.)
struct CopyGuard {
    cudaEvent_t done = nullptr;
    ~CopyGuard() {
        if (!done) return;
        cudaEventSynchronize(done);
        cudaEventDestroy(done);
    }
    cudaError_t copy(void* dst, const void* src, size_t bytes, cudaStream_t st) {
        cudaError_t e = done ? cudaSuccess : cudaEventCreateWithFlags(&done, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
        return e == cudaSuccess ? cudaEventRecord(done, st) : e;
    }
    cudaError_t wait() { return done ? cudaEventSynchronize(done) : cudaSuccess; }
};

double uniform01(uint64_t& s) { return ((splitmix(s) >> 11) + 0.5) * (1.0 / 9007199254740992.0); }

}  // namespace

struct crkdg_mlp {
    unsigned* d_status = nullptr;   // ST_TIMEOUT of a tensor-core wait that ran out
    float* d_prm = nullptr;
    float* d_m = nullptr;
    float* d_v = nullptr;
    float* d_grad = nullptr;
    cudaStream_t stream = nullptr;
    long long adam_t = 0;
    // training workspace, kept between calls: the blocks' gradients and loss
    // sums, the shuffled rows, the minibatches' losses; one call at a time has it
    std::mutex work;
    float* d_gpart = nullptr;
    float* d_lpart = nullptr;
    int* d_idx = nullptr;
    double* d_loss = nullptr;
    size_t part_blocks = 0, idx_cap = 0, loss_cap = 0;
};

// exported for the step kernels' MLP indicator
const float* crkdg_mlp_device_params(const crkdg_mlp* m) { return m ? m->d_prm : nullptr; }

extern "C" {

const char* crkdg_mlp_last_error(void) { return g_merr.c_str(); }

int crkdg_mlp_create(unsigned long long seed, void* stream, crkdg_mlp** out) {
    if (!out) return mfail(CRKDG_EINVAL, "null argument");
    crkdg_mlp* m = new crkdg_mlp();
    m->stream = static_cast<cudaStream_t>(stream);
    std::vector<float> h(MLP_NPARAM, 0.f);
    uint64_t s = seed;
    auto he = [&](int off, int nout, int nin) {
        const double sd = std::sqrt(2.0 / nin);
        for (int i = 0; i < nout * nin; ++i) {
            // Box--Muller normal from two uniforms
            const double u1 = uniform01(s), u2 = uniform01(s);
            h[off + i] = float(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
        }
    };
    he(OW1, MLP_H, MLP_IN);
    he(OW2, MLP_H, MLP_H);
    he(OW3, MLP_H, MLP_H);
    he(OW4, 1, MLP_H);
    if (cudaMalloc(&m->d_prm, MLP_NPARAM * 4) != cudaSuccess || cudaMalloc(&m->d_m, MLP_NPARAM * 4) != cudaSuccess ||
        cudaMalloc(&m->d_v, MLP_NPARAM * 4) != cudaSuccess || cudaMalloc(&m->d_grad, MLP_NPARAM * 4) != cudaSuccess) {
        crkdg_mlp_destroy(m);
        return mfail(CRKDG_ENOMEM, "cudaMalloc failed");
    }
    if (cudaMalloc(&m->d_status, sizeof(unsigned)) != cudaSuccess) {
        crkdg_mlp_destroy(m);
        return mfail(CRKDG_ENOMEM, "cudaMalloc failed");
    }
    cudaMemset(m->d_status, 0, sizeof(unsigned));
    cudaMemcpy(m->d_prm, h.data(), MLP_NPARAM * 4, cudaMemcpyHostToDevice);
    cudaMemset(m->d_m, 0, MLP_NPARAM * 4);
    cudaMemset(m->d_v, 0, MLP_NPARAM * 4);
    *out = m;
    return CRKDG_OK;
}

void crkdg_mlp_destroy(crkdg_mlp* m) {
    if (!m) return;
    cudaStreamSynchronize(m->stream);
    for (float* p : {m->d_prm, m->d_m, m->d_v, m->d_grad})
        if (p) cudaFree(p);
    for (void* p : {(void*)m->d_status, (void*)m->d_gpart, (void*)m->d_lpart, (void*)m->d_idx, (void*)m->d_loss})
        if (p) cudaFree(p);
    delete m;
}

int crkdg_mlp_n_params(void) { return MLP_NPARAM; }

int crkdg_mlp_set_params(crkdg_mlp* m, const float* host) {
    if (!m || !host) return mfail(CRKDG_EINVAL, "null argument");
    MCK(cudaMemcpy(m->d_prm, host, MLP_NPARAM * 4, cudaMemcpyHostToDevice));
    MCK(cudaMemset(m->d_m, 0, MLP_NPARAM * 4));
    MCK(cudaMemset(m->d_v, 0, MLP_NPARAM * 4));
    m->adam_t = 0;
    return CRKDG_OK;
}

int crkdg_mlp_get_params(const crkdg_mlp* m, float* host) {
    if (!m || !host) return mfail(CRKDG_EINVAL, "null argument");
    MCK(cudaStreamSynchronize(m->stream));
    MCK(cudaMemcpy(host, m->d_prm, MLP_NPARAM * 4, cudaMemcpyDeviceToHost));
    return CRKDG_OK;
}

// Blocks of a gradient over n samples: a tile each, one wave at most
static int train_blocks(int n) {
    return (int)std::min<long long>(((long long)n + TILE - 1) / TILE, 2LL * std::max(1, crk::sm_count()));
}

// workspace for gradients over up to n samples and `losses` minibatch losses,
// and the kernel's shared memory
static int train_workspace(crkdg_mlp* m, int n, size_t losses) {
    const size_t blocks = train_blocks(n);
    if (blocks > m->part_blocks) {
        size_t g = m->d_gpart ? m->part_blocks * MLP_NPARAM : 0, l = m->d_lpart ? m->part_blocks : 0;
        m->part_blocks = 0;
        if (!grow(m->d_gpart, g, blocks * MLP_NPARAM) || !grow(m->d_lpart, l, blocks))
            return mfail(CRKDG_ENOMEM, "cudaMalloc failed");
        m->part_blocks = blocks;
    }
    if (!grow(m->d_loss, m->loss_cap, losses)) return mfail(CRKDG_ENOMEM, "cudaMalloc failed");
    // an attribute of the kernel on the current device: set by every call, which
    // may be the device's first
    MCK(cudaFuncSetAttribute(mlp_fwdbwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem)));
    return CRKDG_OK;
}

// Enqueue the mean loss and its gradient over the n samples (rows idx of X, y;
// idx null: in order), *loss and grad on the device, and the Adam step (ad.prm
// null: none).  `follows`: the stream's last work is this function's (X, y and
// idx are read before it has completed).
static cudaError_t enqueue_grad(crkdg_mlp* m, const float* X, const float* y, const int* idx, int n, double pw,
                                double* loss, const AdamArgs& ad, bool follows) {
    const int nb = train_blocks(n);
    const cudaError_t e = launch(&mlp_fwdbwd_kernel, nb, TRAIN_THREADS, sizeof(TrainSmem), follows, m->stream, m->d_prm, X, y,
                                 idx, n, (float)pw, m->d_gpart, m->d_lpart);
    if (e != cudaSuccess) return e;
    return launch(&mlp_reduce_kernel, (MLP_NPARAM + REDUCE_PARAMS - 1) / REDUCE_PARAMS, REDUCE_RUNS * REDUCE_PARAMS, 0, true,
                  m->stream, m->d_gpart, m->d_lpart, nb, n, m->d_grad, loss, ad);
}

int crkdg_mlp_loss_grad(crkdg_mlp* m, const float* X_dev, const float* y_dev, int n, double pos_weight, double* loss,
                        float* grad_host) {
    if (!m || !X_dev || !y_dev || n < 1) return mfail(CRKDG_EINVAL, "bad argument");
    std::lock_guard<std::mutex> own(m->work);
    int r = train_workspace(m, n, 1);
    if (r) return r;
    MCK(enqueue_grad(m, X_dev, y_dev, nullptr, n, pos_weight, m->d_loss, AdamArgs{}, false));
    double l = 0.0;
    MCK(cudaMemcpyAsync(&l, m->d_loss, sizeof l, cudaMemcpyDeviceToHost, m->stream));
    if (grad_host) MCK(cudaMemcpyAsync(grad_host, m->d_grad, MLP_NPARAM * 4, cudaMemcpyDeviceToHost, m->stream));
    MCK(cudaStreamSynchronize(m->stream));
    if (loss) *loss = l;
    return CRKDG_OK;
}

int crkdg_mlp_train(crkdg_mlp* m, const float* X_dev, const float* y_dev, int n, int epochs, int batch, double lr,
                    double pos_weight, unsigned long long seed, double* last_epoch_loss) {
    if (!m || !X_dev || !y_dev || n < 1 || epochs < 0 || batch < 1 || !(lr > 0.0))
        return mfail(CRKDG_EINVAL, "bad argument");
    std::lock_guard<std::mutex> own(m->work);
    const int nb = (int)(((long long)n + batch - 1) / batch);   // minibatches of an epoch
    int r = train_workspace(m, std::min(n, batch), nb);
    if (r) return r;
    if (!grow(m->d_idx, m->idx_cap, n)) return mfail(CRKDG_ENOMEM, "cudaMalloc failed");
    std::vector<int> perm(n);
    for (int i = 0; i < n; ++i) perm[i] = i;
    CopyGuard guard;   // of perm (destroyed before it)
    uint64_t s = seed;
    for (int ep = 0; ep < epochs; ++ep) {
        MCK(guard.wait());   // the last epoch's order has left; its minibatches run on
        for (int i = n - 1; i > 0; --i) {   // Fisher--Yates shuffle
            const int j = (int)(splitmix(s) % (uint64_t)(i + 1));
            std::swap(perm[i], perm[j]);
        }
        MCK(guard.copy(m->d_idx, perm.data(), n * sizeof(int), m->stream));
        for (int b = 0; b < nb; ++b) {
            const int b0 = b * batch, nbatch = std::min(batch, n - b0);
            m->adam_t += 1;
            const float b1 = 0.9f, b2 = 0.999f;
            const float c1 = 1.f - std::pow(b1, (double)m->adam_t), c2 = 1.f - std::pow(b2, (double)m->adam_t);
            const AdamArgs ad{m->d_prm, m->d_m, m->d_v, (float)lr, b1, b2, 1e-8f, c1, c2};
            MCK(enqueue_grad(m, X_dev, y_dev, m->d_idx + b0, nbatch, pos_weight, m->d_loss + b, ad, b > 0));
        }
    }
    double el = 0.0;
    if (epochs > 0) {
        std::vector<double> l(nb);
        MCK(cudaMemcpyAsync(l.data(), m->d_loss, nb * sizeof(double), cudaMemcpyDeviceToHost, m->stream));
        MCK(cudaStreamSynchronize(m->stream));
        for (double v : l) el += v;
        el /= nb;
    }
    MCK(cudaStreamSynchronize(m->stream));
    if (last_epoch_loss) *last_epoch_loss = el;
    return CRKDG_OK;
}

int crkdg_mlp_predict(crkdg_mlp* m, const float* X_dev, int n, float* logits_dev) {
    if (!m || !X_dev || !logits_dev || n < 1) return mfail(CRKDG_EINVAL, "bad argument");
    const size_t smem =
        sizeof(crk::MlpSmem) + (PREDICT_THREADS / 32) * (32 * crk::MLP_INP + 64) * sizeof(__nv_bfloat16);
    auto kern = reinterpret_cast<uintptr_t>(X_dev) % 8 == 0 ? mlp_predict_kernel<true> : mlp_predict_kernel<false>;
    int per_sm = 1;   // (of the current device, as the attribute is)
    MCK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    MCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, PREDICT_THREADS, smem));
    const long long tiles = ((long long)n + PREDICT_THREADS - 1) / PREDICT_THREADS;
    const int grid = (int)std::min<long long>(tiles, (long long)std::max(1, per_sm) * std::max(1, crk::sm_count()));
    kern<<<grid, PREDICT_THREADS, smem, m->stream>>>(m->d_prm, X_dev, n, logits_dev);
    MCK(cudaGetLastError());
    MCK(cudaStreamSynchronize(m->stream));
    return CRKDG_OK;
}

int crkdg_mlp_predict_tc(crkdg_mlp* m, const float* X_dev, int n, float* logits_dev) {
    if (!m || !X_dev || !logits_dev || n < 1) return mfail(CRKDG_EINVAL, "bad argument");
    const size_t smem = sizeof(crk::MlpTcSmem) + crk::MLPTC_SMEM_SLACK;
    MCK(cudaFuncSetAttribute(mlp_predict_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const long long tiles = ((long long)n + crk::MLPTC_CELLS - 1) / crk::MLPTC_CELLS;
    const int grid = (int)std::min<long long>(tiles, 4LL * std::max(1, crk::sm_count()));
    MCK(cudaMemsetAsync(m->d_status, 0, sizeof(unsigned), m->stream));
    mlp_predict_tc_kernel<<<grid, crk::MLPTC_CELLS, smem, m->stream>>>(m->d_prm, X_dev, n, logits_dev, m->d_status);
    MCK(cudaGetLastError());
    unsigned st = 0;
    MCK(cudaMemcpyAsync(&st, m->d_status, sizeof(unsigned), cudaMemcpyDeviceToHost, m->stream));
    MCK(cudaStreamSynchronize(m->stream));
    if (st) return mfail(CRKDG_ETIMEOUT, "a bounded wait for the tensor core ran out");
    return CRKDG_OK;
}

}  // extern "C"

// features of a state slice (used by the context and batch entry points)
int crkdg_features_impl(const StepArgs& a, int precision, int k, int basis, const void* u, float* X, float* y,
                        double Mh2, cudaStream_t st) {
    if (k != 2) return mfail(CRKDG_EUNSUPPORTED, "the learned indicator is built for k = 2");
    StepArgs b = a;
    crk::set_derived(b);
    b.mlp_scale = (float)Mh2;
    const dim3 grid((a.nx + FEAT_THREADS - 1) / FEAT_THREADS, a.ny);
    auto run = [&](auto kern, auto* state) { kern<<<grid, FEAT_THREADS, 0, st>>>(b, state, X, y); };
    const bool P = basis == CRKDG_BASIS_P;
    if (precision == CRKDG_F64)
        run(P ? features_kernel<double, 2, 0> : features_kernel<double, 2, 1>, (const double*)u);
    else
        run(P ? features_kernel<float, 2, 0> : features_kernel<float, 2, 1>, (const float*)u);
    MCK(cudaGetLastError());
    return CRKDG_OK;
}
