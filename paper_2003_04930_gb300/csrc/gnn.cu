// Warm-start network: a 4-layer message-passing network (width 64, BF16
// weights, FP32 accumulation) that predicts the steady-state populations p
// from the graph, so that rho0 = diag(p_hat) starts RK4 near its fixed point.
// Forward, backward and Adam are hand-written kernels; the network is
// trained on steady states the solver itself produces.
//
// Definition (identical to the CPU oracle's, written independently):
//   features x_i = [1, omega, log1p(in-strength), log1p(out-strength),
//                   log1p(in-degree), log1p(out-degree), log(N pi_i), dangles]
//   with A_ij = w for the link j -> i, pi the classical PageRank (stationary
//   vector of G = alpha S + (1 - alpha) F, 200 power-iteration steps from
//   uniform, the omega = 1 limit of the method);
//   P_ij = (A_ij + A_ji) / s_i, s_i = sum_j (A_ij + A_ji);
//   z_l = h_{l-1} Ws_l + (P h_{l-1}) Wn_l + b_l, h_l = relu(z_l), h_0 = x;
//   s = h_4 wo + bo, p_hat = softmax(s), L = -sum_i p_i log p_hat_i.
// The layers are (N x 128) x (128 x 64) products: far too small for tensor
// cores to matter, so they run on the FP32 pipe with the BF16-rounded weights
// staged in shared memory; every reduction (weight gradients, softmax) is in
// fixed order, so training is bitwise reproducible.
#include <limits.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <cstdint>
#include <string>
#include <vector>

#include "qpr_internal.cuh"

namespace qpr {
namespace {

constexpr int FIN = 8, W = 64, LAYERS = 4;
constexpr int kParams = 2 * FIN * W + W + 3 * (2 * W * W + W) + W + 1;  // 25921
constexpr int kRowsWG = 128;  // rows per partial weight-gradient block

// offsets of the flat parameter layout
__host__ __device__ constexpr int off_ws(int l) { return l == 1 ? 0 : 2 * FIN * W + W + (l - 2) * (2 * W * W + W); }
__host__ __device__ constexpr int din_of(int l) { return l == 1 ? FIN : W; }
__host__ __device__ constexpr int off_wn(int l) { return off_ws(l) + din_of(l) * W; }
__host__ __device__ constexpr int off_b(int l) { return off_wn(l) + din_of(l) * W; }
constexpr int OFF_WO = 2 * FIN * W + W + 3 * (2 * W * W + W);
constexpr int OFF_BO = OFF_WO + W;
static_assert(OFF_BO + 1 == kParams, "parameter layout");

// ---------------------------------------------------------------- kernels
// One graph of a group: its arrays and its part of the workspace, on the
// device. Every kernel runs over a group of graphs at once (blockIdx.y is the
// graph): a graph of a few hundred nodes is a few CTAs, and a pass over it is
// a chain of launches, so a mini-batch of eight takes little longer than one.
// Each output is still one sum in the order of a pass over the graph alone,
// and the graphs' gradients are added in the order of the mini-batch.
struct GnnDev {
    int n, nblk;                   // nodes, blocks of kRowsWG rows
    const float *x;                // n x FIN
    const int *pptr, *pcol, *tptr, *tcol;
    const float *pval, *tval;      // P and P^T
    const double *p;               // target populations (or null)
    float *H, *M, *Z;              // per layer 1..4: n x W each (layer l at (l - 1) n W)
    float *dA, *dB, *dT;           // n x W: gradients of a layer's output (alternating) and of P h
    float *s, *ds;                 // n: logits and their gradients
    double *e, *p_hat;             // n
    float *part;                   // nblk x kParams: gradient partials
    double *loss;                  // [0] the graph's loss, [1] log-sum-exp, [2] sum of p
};

// One row of sum_q val[q] X[col[q]][:], d <= 64 columns (lane and lane + 32),
// in entry order. 16 entries' loads are in flight at once: with one at a time
// a hub row of some hundred entries held its launch for 100 us.
__device__ __forceinline__ void row_sum(const int *__restrict__ col, const float *__restrict__ val, int q0, int q1,
                                        const float *__restrict__ X, int d, float &a0, float &a1) {
    constexpr int U = 16;
    const int lane = threadIdx.x & 31;
    const bool c0 = lane < d, c1 = lane + 32 < d;
    a0 = a1 = 0.f;
    for (int qb = q0; qb < q1; qb += 32) {
        const int m = min(32, q1 - qb);
        const int k = lane < m ? col[qb + lane] : 0;
        const float v = lane < m ? val[qb + lane] : 0.f;
        for (int e = 0; e < m; e += U) {
            float x0[U], x1[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float *x = X + (size_t)__shfl_sync(0xffffffffu, k, (e + u) & 31) * d + lane;
                const bool on = e + u < m;
                x0[u] = on && c0 ? x[0] : 0.f;
                x1[u] = on && c1 ? x[32] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float vu = __shfl_sync(0xffffffffu, v, (e + u) & 31);
                if (e + u < m) {  // uniform: adding 0 could turn -0 into 0
                    a0 = __fmaf_rn(vu, x0[u], a0);
                    a1 = __fmaf_rn(vu, x1[u], a1);
                }
            }
        }
    }
}

// Layer l of 8 rows per CTA: M = P h, Z = h Ws + M Wn + b, H = relu(Z); the
// last layer also forms the logits s = H wo + bo.
constexpr int kFwdRows = 8;
__global__ void __launch_bounds__(256) layer_fwd_kernel(const GnnDev *__restrict__ gs, const float *__restrict__ prm,
                                                        int l) {
    __shared__ float sW[2 * W * W];
    __shared__ float sH[kFwdRows * W], sM[kFwdRows * W], sO[kFwdRows * W];
    const GnnDev g = gs[blockIdx.y];
    const int n = g.n, r0 = blockIdx.x * kFwdRows;
    if (r0 >= n) return;
    const int din = din_of(l), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t nw = (size_t)n * W;
    const float *h = l == 1 ? g.x : g.H + (l - 2) * nw;
    for (int t = threadIdx.x; t < 2 * din * W; t += blockDim.x) sW[t] = prm[off_ws(l) + t];  // Ws then Wn
    for (int t = threadIdx.x; t < kFwdRows * din; t += blockDim.x) {
        const int r = r0 + t / din;
        sH[t] = r < n ? h[(size_t)r * din + t % din] : 0.f;
    }
    {
        const int r = r0 + warp;
        float a0 = 0.f, a1 = 0.f;
        if (r < n) {
            row_sum(g.pcol, g.pval, g.pptr[r], g.pptr[r + 1], h, din, a0, a1);
            float *m = g.M + (l - 1) * nw + (size_t)r * din;
            if (lane < din) m[lane] = a0;
            if (lane + 32 < din) m[lane + 32] = a1;
        }
        if (lane < din) sM[warp * din + lane] = a0;
        if (lane + 32 < din) sM[warp * din + lane + 32] = a1;
    }
    __syncthreads();
    const int f = threadIdx.x & (W - 1), q = threadIdx.x >> 6;  // rows q and q + 4
    const float bf = prm[off_b(l) + f];
    float z0 = bf, z1 = bf;
    for (int k = 0; k < din; ++k) {
        const float ws = sW[k * W + f], wn = sW[din * W + k * W + f];
        z0 = __fmaf_rn(sH[q * din + k], ws, z0);
        z1 = __fmaf_rn(sH[(q + 4) * din + k], ws, z1);
        z0 = __fmaf_rn(sM[q * din + k], wn, z0);
        z1 = __fmaf_rn(sM[(q + 4) * din + k], wn, z1);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int rr = q + 4 * j, r = r0 + rr;
        const float z = j ? z1 : z0, o = z > 0.f ? z : 0.f;
        sO[rr * W + f] = o;
        if (r < n) {
            g.Z[(l - 1) * nw + (size_t)r * W + f] = z;
            g.H[(l - 1) * nw + (size_t)r * W + f] = o;
        }
    }
    if (l < LAYERS) return;
    __syncthreads();
    if (threadIdx.x < kFwdRows && r0 + (int)threadIdx.x < n) {
        float s = prm[OFF_BO];
        for (int k = 0; k < W; ++k) s = __fmaf_rn(sO[threadIdx.x * W + k], prm[OFF_WO + k], s);
        g.s[r0 + threadIdx.x] = s;
    }
}

// Softmax and loss of a graph by a cluster of 8 CTAs: p_hat = softmax(s); L =
// -sum p_i log p_hat_i; ds_i = p_hat_i sum(p) - p_i. The exponentials are FP64
// (some 25 instructions, 40 ns each per scheduler: 38 us in one CTA at N =
// 1000), so the CTAs share them; the first one forms the sums, in a fixed
// order (its 256 threads over i, i + 256, ..., then the warps).
constexpr int kSoftCtas = 8;
__global__ void __cluster_dims__(kSoftCtas, 1, 1) __launch_bounds__(256)
softmax_loss_kernel(const GnnDev *__restrict__ gs) {
    __shared__ double red[8];
    __shared__ float redf[8];
    __shared__ double bc;
    const GnnDev g = gs[blockIdx.y];
    const int n = g.n, cta = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float *__restrict__ sb = g.s;
    const double *__restrict__ p = g.p;
    auto bsum = [&](double v) {
        for (int o = 16; o > 0; o >>= 1) v = v + __shfl_xor_sync(0xffffffffu, v, o);
        __syncthreads();
        if (lane == 0) red[warp] = v;
        __syncthreads();
        if (tid == 0) {
            double t = red[0];
            for (int q = 1; q < 8; ++q) t = t + red[q];
            bc = t;
        }
        __syncthreads();
        return bc;
    };
    auto barrier = [] {
        __syncthreads();
        asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    };
    float mf = -INFINITY;
    for (int i = tid; i < n; i += 256) mf = fmaxf(mf, sb[i]);
    for (int o = 16; o > 0; o >>= 1) mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
    if (lane == 0) redf[warp] = mf;
    __syncthreads();
    for (int q = 0; q < 8; ++q) mf = fmaxf(mf, redf[q]);
    const double mx = (double)mf;
    for (int i = cta * 256 + tid; i < n; i += kSoftCtas * 256) g.e[i] = exp((double)sb[i] - mx);
    barrier();
    if (cta == 0) {
        double se = 0.0, sp = 0.0;
        for (int i = tid; i < n; i += 256) {
            se += __ldcg(g.e + i);
            sp += p ? p[i] : 0.0;
        }
        se = bsum(se);
        sp = bsum(sp);
        if (tid == 0) {
            g.loss[1] = mx + log(se);
            g.loss[2] = sp;
        }
    }
    barrier();
    const double lse = __ldcg(g.loss + 1), sp = __ldcg(g.loss + 2);
    for (int i = cta * 256 + tid; i < n; i += kSoftCtas * 256) {
        const double ph = exp((double)sb[i] - lse);
        g.p_hat[i] = ph;
        if (p) g.ds[i] = (float)(ph * sp - p[i]);
    }
    if (p && cta == 0) {
        double ls = 0.0;
        for (int i = tid; i < n; i += 256) {
            const double lp = (double)sb[i] - lse;
            ls -= p[i] * lp;
        }
        ls = bsum(ls);
        if (tid == 0) g.loss[0] = ls;
    }
}

// dH4 = ds wo^T (n x 64), and the partial sums of dwo = H4^T ds, dbo = sum ds
// per block of kRowsWG rows (staged in shared memory: the sums run over rows).
__global__ void __launch_bounds__(256) readout_bwd_kernel(const GnnDev *__restrict__ gs, const float *__restrict__ prm) {
    __shared__ float sH[kRowsWG * W];
    __shared__ float sd[kRowsWG];
    const GnnDev g = gs[blockIdx.y];
    if ((int)blockIdx.x >= g.nblk) return;
    const int r0 = blockIdx.x * kRowsWG, rows = min(g.n - r0, kRowsWG);
    const float *H4 = g.H + (size_t)(LAYERS - 1) * g.n * W;
    for (int t = threadIdx.x; t < rows; t += blockDim.x) sd[t] = g.ds[r0 + t];
    for (int t = threadIdx.x; t < rows * W; t += blockDim.x) sH[t] = H4[(size_t)r0 * W + t];
    __syncthreads();
    float *part = g.part + (size_t)blockIdx.x * kParams + OFF_WO;
    if (threadIdx.x < W) {
        float gw = 0.f;
        for (int r = 0; r < rows; ++r) gw = __fmaf_rn(sH[r * W + threadIdx.x], sd[r], gw);
        part[threadIdx.x] = gw;
    } else if (threadIdx.x == W) {
        float gb = 0.f;
        for (int r = 0; r < rows; ++r) gb = __fadd_rn(gb, sd[r]);
        part[W] = gb;
    }
    const float wo = prm[OFF_WO + (threadIdx.x & (W - 1))];
    for (int t = threadIdx.x; t < rows * W; t += blockDim.x) g.dA[(size_t)r0 * W + t] = __fmul_rn(sd[t / W], wo);
}

// Partial sums of dWs = h^T dZ, dWn = M^T dZ, db = sum dZ of layer l per block
// of kRowsWG rows, dZ = dH [Z > 0]. A CTA takes kWgCols columns of [h | M] (16
// CTAs a block at width 64; one CTA a block left 8 of them on the chip at N =
// 1000, 90 us) with the block's rows in shared memory.
constexpr int kWgCols = 8;
__global__ void __launch_bounds__(256) wgrad_kernel(const GnnDev *__restrict__ gs, int l, int odd) {
    __shared__ float sdz[kRowsWG * W];
    __shared__ float src[kRowsWG * kWgCols];
    const GnnDev g = gs[blockIdx.y];
    const int din = din_of(l), splits = 2 * din / kWgCols;
    const int blk = blockIdx.x / splits, c0 = (blockIdx.x - blk * splits) * kWgCols;
    if (blk >= g.nblk) return;
    const int n = g.n, r0 = blk * kRowsWG, rows = min(n - r0, kRowsWG);
    const size_t nw = (size_t)n * W;
    const float *h = l == 1 ? g.x : g.H + (l - 2) * nw, *M = g.M + (l - 1) * nw, *Z = g.Z + (l - 1) * nw;
    const float *dH = odd ? g.dB : g.dA;
    for (int t = threadIdx.x; t < rows * W; t += blockDim.x) {
        const size_t o = (size_t)r0 * W + t;
        sdz[t] = Z[o] > 0.f ? dH[o] : 0.f;
    }
    for (int t = threadIdx.x; t < rows * kWgCols; t += blockDim.x) {
        const int rr = t / kWgCols, c = c0 + t % kWgCols;
        src[t] = (c < din ? h : M)[(size_t)(r0 + rr) * din + (c < din ? c : c - din)];
    }
    __syncthreads();
    const int f = threadIdx.x & (W - 1), k = threadIdx.x >> 6;  // columns k and k + 4
    float a0 = 0.f, a1 = 0.f;
    for (int rr = 0; rr < rows; ++rr) {
        const float dz = sdz[rr * W + f];
        a0 = __fmaf_rn(src[rr * kWgCols + k], dz, a0);
        a1 = __fmaf_rn(src[rr * kWgCols + k + 4], dz, a1);
    }
    float *out = g.part + (size_t)blk * kParams + off_ws(l);
    out[(c0 + k) * W + f] = a0;
    out[(c0 + k + 4) * W + f] = a1;
    if (c0 == 0 && k == 0) {
        float b = 0.f;
        for (int rr = 0; rr < rows; ++rr) b = __fadd_rn(b, sdz[rr * W + f]);
        out[2 * din * W + f] = b;
    }
}

// dHs = dZ Ws^T, dT = dZ Wn^T of layer l >= 2 (n x 64), dZ = dH [Z > 0]: 8
// rows per CTA, the weights in shared memory (rows padded: the lanes read a
// column).
__global__ void __launch_bounds__(256) dense_bwd_kernel(const GnnDev *__restrict__ gs, const float *__restrict__ prm,
                                                        int l, int odd) {
    constexpr int LD = W + 1;
    __shared__ float sS[W * LD], sN[W * LD], sdz[kFwdRows * W];
    const GnnDev g = gs[blockIdx.y];
    const int n = g.n, r0 = blockIdx.x * kFwdRows;
    if (r0 >= n) return;
    const float *dH = odd ? g.dB : g.dA;
    float *dHs = odd ? g.dA : g.dB;
    const float *Z = g.Z + (size_t)(l - 1) * n * W;
    for (int t = threadIdx.x; t < W * W; t += blockDim.x) {
        sS[(t / W) * LD + t % W] = prm[off_ws(l) + t];
        sN[(t / W) * LD + t % W] = prm[off_wn(l) + t];
    }
    for (int t = threadIdx.x; t < kFwdRows * W; t += blockDim.x) {
        const size_t o = (size_t)r0 * W + t;
        sdz[t] = r0 + t / W < n && Z[o] > 0.f ? dH[o] : 0.f;
    }
    __syncthreads();
    const int k = threadIdx.x & (W - 1), q = threadIdx.x >> 6;
    float a0 = 0.f, b0 = 0.f, a1 = 0.f, b1 = 0.f;
    for (int f = 0; f < W; ++f) {
        const float ws = sS[k * LD + f], wn = sN[k * LD + f], d0 = sdz[q * W + f], d1 = sdz[(q + 4) * W + f];
        a0 = __fmaf_rn(d0, ws, a0);
        b0 = __fmaf_rn(d0, wn, b0);
        a1 = __fmaf_rn(d1, ws, a1);
        b1 = __fmaf_rn(d1, wn, b1);
    }
    if (r0 + q < n) {
        dHs[(size_t)(r0 + q) * W + k] = a0;
        g.dT[(size_t)(r0 + q) * W + k] = b0;
    }
    if (r0 + q + 4 < n) {
        dHs[(size_t)(r0 + q + 4) * W + k] = a1;
        g.dT[(size_t)(r0 + q + 4) * W + k] = b1;
    }
}

// dH of the layer below = dHs + P^T dT, one warp per row.
__global__ void __launch_bounds__(256) spmm_bwd_kernel(const GnnDev *__restrict__ gs, int odd) {
    const GnnDev g = gs[blockIdx.y];
    const int lane = threadIdx.x & 31, i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= g.n) return;
    float a0, a1;
    row_sum(g.tcol, g.tval, g.tptr[i], g.tptr[i + 1], g.dT, W, a0, a1);
    float *y = (odd ? g.dA : g.dB) + (size_t)i * W;
    y[lane] = __fadd_rn(y[lane], a0);
    y[lane + 32] = __fadd_rn(y[lane + 32], a1);
}

// grad (zero first with `init`) += each graph's gradient (its blocks' partials
// in order), graph after graph; *loss likewise.
__global__ void reduce_kernel(const GnnDev *__restrict__ gs, int count, int init, float *__restrict__ grad,
                              double *__restrict__ loss) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) {
        double l = *loss;
        for (int k = 0; k < count; ++k) l += gs[k].loss[0];
        *loss = l;
    }
    if (t >= kParams) return;
    float acc = init ? 0.f : grad[t];
    for (int k = 0; k < count; ++k) {
        const float *part = gs[k].part;
        const int nblk = gs[k].nblk;
        float s = 0.f;
#pragma unroll 4
        for (int b = 0; b < nblk; ++b) s = __fadd_rn(s, part[(size_t)b * kParams + t]);
        acc = __fadd_rn(acc, s);
    }
    grad[t] = acc;
}

// Adam (bias-corrected) on the FP32 master weights; the forward copy keeps
// the weight matrices rounded to BF16 and the biases as stored.
__global__ void adam_kernel(float *__restrict__ theta, float *__restrict__ fwd, const float *__restrict__ grad,
                            float *__restrict__ m, float *__restrict__ v, float inv_batch, float lr, float b1,
                            float b2, float eps, float c1, float c2, int n) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const float g = grad[t] * inv_batch;
    const float mt = b1 * m[t] + (1.f - b1) * g;
    const float vt = b2 * v[t] + (1.f - b2) * g * g;
    m[t] = mt;
    v[t] = vt;
    const float th = theta[t] - lr * (mt / c1) / (sqrtf(vt / c2) + eps);
    theta[t] = th;
    bool is_w = false;
    for (int l = 1; l <= LAYERS; ++l)
        if (t >= off_ws(l) && t < off_b(l)) is_w = true;
    fwd[t] = is_w ? __bfloat162float(__float2bfloat16_rn(th)) : th;
}

__global__ void round_params_kernel(const float *__restrict__ theta, float *__restrict__ fwd, int n) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    bool is_w = false;
    for (int l = 1; l <= LAYERS; ++l)
        if (t >= off_ws(l) && t < off_b(l)) is_w = true;
    fwd[t] = is_w ? __bfloat162float(__float2bfloat16_rn(theta[t])) : theta[t];
}

// ---------------------------------------------------------------- host side
struct HostGraph {
    int n = 0;
    std::vector<float> x;                        // n x FIN
    std::vector<int> pptr, pcol, tptr, tcol;     // P and P^T in CSR
    std::vector<float> pval, tval;
    // the PageRank feature (x_6) is formed on the device from these (up to
    // kPrClusterMaxN nodes; above, here)
    bool device_pr = false;
    double alpha = 0.0;
    std::vector<int> sptr, scol;
    std::vector<double> sval;
    std::vector<unsigned char> dang;
};

constexpr int kPrIters = 200, kPrFeature = 6;

// Below this many entries and nodes a lone graph's power iteration is faster
// here (measured: N = 100 230 us a call, N = 200 470) than in a cluster (3 us an iteration
// whatever the graph: N = 130 to 200 540 to 610); the graphs of a training set run
// side by side there.
constexpr int kPrHostWork = 2200;

// Features and aggregation of one graph (see the file header); one of many?
qpr_status build_graph(int64_t n, int64_t m, const int64_t *src, const int64_t *dst, const double *w, double alpha,
                       double omega, HostGraph &out, std::string &err, bool many = false) {
    HostOps h;
    const qpr_status st = assemble_host(n, m, src, dst, w, QPR_HDIAG_ZERO, h, err, false);
    if (st != QPR_OK) return st;
    // A entries (i, j, a) from the CSR of S: A_ij = S_ij outDeg(j); and of
    // the transpose, columns in order
    const size_t nnz = h.scol.size();
    std::vector<double> av(nnz), tv(nnz);
    std::vector<int> tp(n + 1, 0), tc(nnz);
    std::vector<double> instr(n, 0.0);
    for (int64_t i = 0; i < n; ++i)
        for (int q = h.sptr[i]; q < h.sptr[i + 1]; ++q) {
            av[q] = h.sval[q] * h.outdeg[h.scol[q]];
            instr[i] += av[q];
            tp[h.scol[q] + 1] += 1;
        }
    for (int64_t i = 0; i < n; ++i) tp[i + 1] += tp[i];
    {
        std::vector<int> at(tp.begin(), tp.end() - 1);
        for (int64_t i = 0; i < n; ++i)
            for (int q = h.sptr[i]; q < h.sptr[i + 1]; ++q) {
                const int t = at[h.scol[q]]++;
                tc[t] = (int)i;
                tv[t] = av[q];
            }
    }
    out.n = (int)n;
    out.x.assign((size_t)n * FIN, 0.f);
    for (int64_t i = 0; i < n; ++i) {
        float *x = &out.x[(size_t)i * FIN];
        x[0] = 1.f;
        x[1] = (float)omega;
        x[2] = (float)log1p(instr[i]);
        x[3] = (float)log1p(h.outdeg[i]);
        x[4] = (float)log1p((double)(h.sptr[i + 1] - h.sptr[i]));
        x[5] = (float)log1p((double)(tp[i + 1] - tp[i]));
        x[7] = h.dang[i] ? 1.f : 0.f;
    }
    // B = A + A^T row by row (the two sorted rows merged), P = B
    // row-normalised; B is symmetric, so P^T has its pattern
    out.pptr.assign(n + 1, 0);
    out.pcol.reserve(2 * nnz);
    std::vector<double> bv, rs(n, 0.0);
    bv.reserve(2 * nnz);
    for (int64_t i = 0; i < n; ++i) {
        int qa = h.sptr[i], qt = tp[i];
        while (qa < h.sptr[i + 1] || qt < tp[i + 1]) {
            const int ja = qa < h.sptr[i + 1] ? h.scol[qa] : INT_MAX, jt = qt < tp[i + 1] ? tc[qt] : INT_MAX;
            const int j = std::min(ja, jt);
            double v = 0.0;
            if (ja == j) v = av[qa++];
            if (jt == j) v += tv[qt++];
            out.pcol.push_back(j);
            bv.push_back(v);
            rs[i] += v;
        }
        out.pptr[i + 1] = (int)out.pcol.size();
    }
    out.tptr = out.pptr;
    out.tcol = out.pcol;
    out.pval.resize(bv.size());
    out.tval.resize(bv.size());
    for (int64_t i = 0; i < n; ++i)
        for (int q = out.pptr[i]; q < out.pptr[i + 1]; ++q) {
            out.pval[q] = (float)(bv[q] / rs[i]);
            out.tval[q] = (float)(bv[q] / rs[out.pcol[q]]);
        }
    out.device_pr = n <= kPrClusterMaxN && (many || (int64_t)nnz + 2 * n > kPrHostWork);
    out.alpha = alpha;
    if (out.device_pr) {
        out.sptr = std::move(h.sptr);
        out.scol = std::move(h.scol);
        out.sval = std::move(h.sval);
        out.dang = std::move(h.dang);
        return QPR_OK;
    }
    // classical PageRank: pi <- G pi, renormalised, 200 steps from uniform
    std::vector<double> pi(n, 1.0 / (double)n), nx(n);
    const double inv_nm1 = 1.0 / (double)(n - 1);
    for (int it = 0; it < kPrIters; ++it) {
        double P = 0.0, D = 0.0;
        for (int64_t j = 0; j < n; ++j) {
            P += pi[j];
            if (h.dang[j]) D += pi[j];
        }
        double tot = 0.0;
        for (int64_t i = 0; i < n; ++i) {
            double s = 0.0;
            for (int q = h.sptr[i]; q < h.sptr[i + 1]; ++q) s += h.sval[q] * pi[h.scol[q]];
            const double dterm = (D - (h.dang[i] ? pi[i] : 0.0)) * inv_nm1;
            nx[i] = alpha * (s + dterm) + (1.0 - alpha) * (P - pi[i]) * inv_nm1;
            tot += nx[i];
        }
        for (int64_t i = 0; i < n; ++i) pi[i] = nx[i] / tot;
    }
    for (int64_t i = 0; i < n; ++i) out.x[(size_t)i * FIN + kPrFeature] = (float)log((double)n * pi[i]);
    return QPR_OK;
}

uint64_t splitmix(uint64_t &s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

}  // namespace
}  // namespace qpr

struct qpr_gnn {
    int device = 0;
    cudaStream_t stream = nullptr;
    float *theta = nullptr, *fwd = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    int64_t adam_t = 0;
    // device memory grown on demand: the graphs, the group's descriptors, the
    // workspace (sized in nodes and blocks of a group)
    char *graphs = nullptr, *ws = nullptr;
    size_t graphs_cap = 0, ws_cap = 0;
    qpr::GnnDev *desc = nullptr;  // pinned: descriptors of the groups in flight
    size_t desc_cap = 0;
    double *loss = nullptr;
    std::vector<void *> bufs;
    std::string err;
};

namespace {

using qpr::FIN;
using qpr::W;

qpr_status gnn_fail(qpr_gnn *g, qpr_status st, const std::string &msg) {
    if (g) g->err = msg;
    qpr::set_create_error(msg);
    return st;
}

#define GCUDA(g, call)                                                                                     \
    do {                                                                                                   \
        cudaError_t e_ = (call);                                                                           \
        if (e_ != cudaSuccess)                                                                             \
            return gnn_fail(g, e_ == cudaErrorMemoryAllocation ? QPR_E_OOM : QPR_E_CUDA,                   \
                            std::string(#call) + ": " + cudaGetErrorString(e_));                           \
    } while (0)

template <class T>
cudaError_t galloc(qpr_gnn *g, T **p, size_t count) {
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, std::max<size_t>(count, 1) * sizeof(T));
    if (e == cudaSuccess) {
        g->bufs.push_back(q);
        *p = (T *)q;
    }
    return e;
}

size_t round16(size_t b) { return (b + 15) & ~(size_t)15; }

// Grow *buf to `bytes`.
qpr_status grow(qpr_gnn *g, char **buf, size_t *cap, size_t bytes) {
    if (bytes <= *cap) return QPR_OK;
    if (*buf) {
        GCUDA(g, cudaStreamSynchronize(g->stream));
        cudaFree(*buf);
        *buf = nullptr;
        *cap = 0;
    }
    GCUDA(g, cudaMalloc((void **)buf, bytes));
    *cap = bytes;
    return QPR_OK;
}

// Bytes of a graph in device memory (with what its PageRank feature is
// formed from, until it has one), and the image of it with the pointers that
// it has at `dev`; a PageRank job goes to `jobs`.
size_t graph_bytes(const qpr::HostGraph &hg) {
    const size_t n = hg.n, nnz = hg.pcol.size();
    size_t b = round16(hg.x.size() * 4) + 2 * round16((n + 1) * 4) + 4 * round16(nnz * 4) + round16(n * 8);
    if (hg.device_pr) b += round16((n + 1) * 4) + round16(hg.scol.size() * 4) + round16(hg.sval.size() * 8) + round16(n);
    return b;
}
void put_graph(const qpr::HostGraph &hg, const double *p, char *host, char *dev, qpr::GnnDev *d,
               std::vector<qpr::PrJob> &jobs) {
    size_t at = 0;
    auto put = [&](const void *src, size_t bytes) {
        if (bytes) memcpy(host + at, src, bytes);
        char *q = dev + at;
        at += round16(bytes);
        return q;
    };
    d->n = hg.n;
    d->nblk = (hg.n + qpr::kRowsWG - 1) / qpr::kRowsWG;
    d->x = (const float *)put(hg.x.data(), hg.x.size() * 4);
    d->pptr = (const int *)put(hg.pptr.data(), hg.pptr.size() * 4);
    d->tptr = (const int *)put(hg.tptr.data(), hg.tptr.size() * 4);
    d->pcol = (const int *)put(hg.pcol.data(), hg.pcol.size() * 4);
    d->tcol = (const int *)put(hg.tcol.data(), hg.tcol.size() * 4);
    d->pval = (const float *)put(hg.pval.data(), hg.pval.size() * 4);
    d->tval = (const float *)put(hg.tval.data(), hg.tval.size() * 4);
    d->p = p ? (const double *)put(p, (size_t)hg.n * 8) : nullptr;
    if (!hg.device_pr) return;
    qpr::PrJob j{};
    j.n = hg.n;
    j.dangling = QPR_DANGLING_F;
    j.alpha = hg.alpha;
    j.s_ptr = (const int *)put(hg.sptr.data(), hg.sptr.size() * 4);
    j.s_col = (const int *)put(hg.scol.data(), hg.scol.size() * 4);
    j.s_val = (const double *)put(hg.sval.data(), hg.sval.size() * 8);
    j.dang = (const unsigned char *)put(hg.dang.data(), hg.dang.size());
    j.feature = const_cast<float *>(d->x) + qpr::kPrFeature;
    j.stride = qpr::FIN;
    jobs.push_back(j);
}

// Upload graphs (targets p[i], or null) into g->graphs, their descriptors to
// graphs[i], and form the PageRank features of those that have none. Returns
// with `img` free again.
qpr_status upload_graphs(qpr_gnn *g, const std::vector<const qpr::HostGraph *> &hg, const std::vector<const double *> &p,
                         const std::vector<qpr::GnnDev *> &graphs, std::vector<char> &img) {
    size_t bytes = 0;
    int maxn = 0;
    for (const qpr::HostGraph *h : hg) {
        bytes += graph_bytes(*h);
        if (h->device_pr) maxn = std::max(maxn, h->n);
    }
    const size_t all = bytes + hg.size() * sizeof(qpr::PrJob);
    const qpr_status st = grow(g, &g->graphs, &g->graphs_cap, all);
    if (st != QPR_OK) return st;
    if (img.size() < all) img.resize(all);
    std::vector<qpr::PrJob> jobs;
    size_t at = 0;
    for (size_t k = 0; k < hg.size(); ++k) {
        put_graph(*hg[k], p[k], img.data() + at, g->graphs + at, graphs[k], jobs);
        at += graph_bytes(*hg[k]);
    }
    if (!jobs.empty()) memcpy(img.data() + bytes, jobs.data(), jobs.size() * sizeof(qpr::PrJob));
    GCUDA(g, cudaMemcpyAsync(g->graphs, img.data(), bytes + jobs.size() * sizeof(qpr::PrJob), cudaMemcpyHostToDevice,
                             g->stream));
    if (!jobs.empty())
        GCUDA(g, qpr::pagerank_jobs((const qpr::PrJob *)(g->graphs + bytes), (int)jobs.size(), maxn, qpr::kPrIters,
                                    g->stream));
    GCUDA(g, cudaStreamSynchronize(g->stream));
    return QPR_OK;
}

// Bytes of workspace of one graph.
size_t ws_bytes(int n) {
    const size_t nw = (size_t)n * W, nblk = (n + qpr::kRowsWG - 1) / qpr::kRowsWG;
    return round16((15 * nw + 2 * (size_t)n) * 4) + 2 * round16((size_t)n * 8) + round16(nblk * qpr::kParams * 4) + 32;
}
void place_ws(char *at, qpr::GnnDev *d) {
    const size_t n = d->n, nw = n * W;
    float *f = (float *)at;
    d->H = f;
    d->M = f + 4 * nw;
    d->Z = f + 8 * nw;
    d->dA = f + 12 * nw;
    d->dB = f + 13 * nw;
    d->dT = f + 14 * nw;
    d->s = f + 15 * nw;
    d->ds = d->s + n;
    at += round16((15 * nw + 2 * n) * 4);
    d->e = (double *)at;
    at += round16(n * 8);
    d->p_hat = (double *)at;
    at += round16(n * 8);
    d->part = (float *)at;
    at += round16((size_t)d->nblk * qpr::kParams * 4);
    d->loss = (double *)at;
}

// Room for `count` pinned descriptors.
qpr_status grow_desc(qpr_gnn *g, size_t count) {
    if (count <= g->desc_cap) return QPR_OK;
    GCUDA(g, cudaStreamSynchronize(g->stream));
    cudaFreeHost(g->desc);
    g->desc = nullptr;
    g->desc_cap = 0;
    GCUDA(g, cudaMallocHost((void **)&g->desc, count * sizeof(qpr::GnnDev)));
    g->desc_cap = count;
    return QPR_OK;
}

// The workspace of a group (count descriptors at grp, pinned and left alone
// until the stream has been waited for) and its descriptors behind it on the
// device.
qpr_status place_group(qpr_gnn *g, qpr::GnnDev *grp, size_t count, qpr::GnnDev **dev) {
    size_t bytes = 0;
    for (size_t k = 0; k < count; ++k) bytes += ws_bytes(grp[k].n);
    const qpr_status st = grow(g, &g->ws, &g->ws_cap, bytes + count * sizeof(qpr::GnnDev));
    if (st != QPR_OK) return st;
    size_t at = 0;
    for (size_t k = 0; k < count; ++k) {
        place_ws(g->ws + at, &grp[k]);
        at += ws_bytes(grp[k].n);
    }
    *dev = (qpr::GnnDev *)(g->ws + at);
    GCUDA(g, cudaMemcpyAsync(*dev, grp, count * sizeof(qpr::GnnDev), cudaMemcpyHostToDevice, g->stream));
    return QPR_OK;
}

// Forward pass of a group (and, with targets, loss and backward into g->grad,
// zeroed first with `init`).
void enqueue_pass(qpr_gnn *g, const qpr::GnnDev *dev, int count, int maxn, bool backward, bool init) {
    cudaStream_t s = g->stream;
    const dim3 rows((maxn + qpr::kFwdRows - 1) / qpr::kFwdRows, count);
    for (int l = 1; l <= qpr::LAYERS; ++l) qpr::layer_fwd_kernel<<<rows, 256, 0, s>>>(dev, g->fwd, l);
    qpr::softmax_loss_kernel<<<dim3(qpr::kSoftCtas, count), 256, 0, s>>>(dev);
    if (!backward) return;
    const int nblk = (maxn + qpr::kRowsWG - 1) / qpr::kRowsWG;
    qpr::readout_bwd_kernel<<<dim3(nblk, count), 256, 0, s>>>(dev, g->fwd);
    int odd = 0;  // the output gradient of the layer is in dB
    for (int l = qpr::LAYERS; l >= 1; --l) {
        const int splits = 2 * qpr::din_of(l) / qpr::kWgCols;
        qpr::wgrad_kernel<<<dim3(nblk * splits, count), 256, 0, s>>>(dev, l, odd);
        if (l > 1) {
            qpr::dense_bwd_kernel<<<rows, 256, 0, s>>>(dev, g->fwd, l, odd);
            qpr::spmm_bwd_kernel<<<dim3((maxn + 7) / 8, count), 256, 0, s>>>(dev, odd);
            odd ^= 1;
        }
    }
    qpr::reduce_kernel<<<(qpr::kParams + 127) / 128, 128, 0, s>>>(dev, count, init ? 1 : 0, g->grad, g->loss);
}

// One graph, as predict and loss_grad run it.
qpr_status single_pass(qpr_gnn *g, const qpr::HostGraph &hg, const double *p, bool backward, qpr::GnnDev *out) {
    qpr_status st = grow_desc(g, 1);
    if (st != QPR_OK) return st;
    std::vector<char> img;
    st = upload_graphs(g, {&hg}, {p}, {g->desc}, img);
    if (st != QPR_OK) return st;
    qpr::GnnDev *dev = nullptr;
    st = place_group(g, g->desc, 1, &dev);
    if (st != QPR_OK) return st;
    if (backward) GCUDA(g, cudaMemsetAsync(g->loss, 0, sizeof(double), g->stream));
    enqueue_pass(g, dev, 1, hg.n, backward, true);
    *out = g->desc[0];
    // the descriptor is free again after this
    GCUDA(g, cudaStreamSynchronize(g->stream));
    return QPR_OK;
}

// Workspace of a group at most (unless one graph needs more): some 70,000 nodes
// in graphs of hundreds (4.7 KB a node), 2000 graphs of a few nodes (a block of
// 128 rows of partial gradients, 104 KB, for the smallest).
constexpr size_t kGroupBytes = (size_t)320 << 20;
// The training set stays on the device up to this size; beyond it every group
// is uploaded for its pass.
constexpr size_t kResidentBytes = (size_t)2 << 30;

}  // namespace

extern "C" {

int64_t qpr_gnn_param_count(void) { return qpr::kParams; }

void qpr_gnn_destroy(qpr_gnn *g) {
    if (!g) return;
    int prev = -1;
    cudaGetDevice(&prev);
    cudaSetDevice(g->device);
    if (g->stream) cudaStreamSynchronize(g->stream);
    for (void *p : g->bufs) cudaFree(p);
    cudaFree(g->graphs);
    cudaFree(g->ws);
    cudaFreeHost(g->desc);
    if (g->stream) cudaStreamDestroy(g->stream);
    cudaGetLastError();
    if (prev >= 0) cudaSetDevice(prev);
    delete g;
}

qpr_status qpr_gnn_create(qpr_gnn **out, uint64_t seed, int32_t device) {
    if (!out) return QPR_E_ARG;
    *out = nullptr;
    qpr_gnn *g = new (std::nothrow) qpr_gnn();
    if (!g) return gnn_fail(nullptr, QPR_E_OOM, "host allocation failed");
    if (device < 0) {
        if (cudaGetDevice(&g->device) != cudaSuccess) {
            cudaGetLastError();
            delete g;
            return gnn_fail(nullptr, QPR_E_CUDA, "no CUDA device available");
        }
    } else {
        g->device = device;
    }
    cudaSetDevice(g->device);
    auto bail = [&](qpr_status st) {
        qpr_gnn_destroy(g);
        return st;
    };
    const int P = qpr::kParams;
    if (galloc(g, &g->theta, P) != cudaSuccess || galloc(g, &g->fwd, P) != cudaSuccess ||
        galloc(g, &g->grad, P) != cudaSuccess || galloc(g, &g->m, P) != cudaSuccess ||
        galloc(g, &g->v, P) != cudaSuccess || galloc(g, &g->loss, 1) != cudaSuccess || cudaStreamCreateWithFlags(&g->stream, cudaStreamNonBlocking) != cudaSuccess)
        return bail(gnn_fail(nullptr, QPR_E_OOM, "device allocation failed"));
    // Glorot-uniform weights from splitmix64(seed), zero biases
    std::vector<float> th(P, 0.f);
    uint64_t st = seed;
    for (int l = 1; l <= qpr::LAYERS; ++l) {
        const int din = qpr::din_of(l);
        const double lim = sqrt(6.0 / (double)(2 * din + W));
        for (int t = qpr::off_ws(l); t < qpr::off_b(l); ++t)
            th[t] = (float)(lim * (2.0 * ((double)(qpr::splitmix(st) >> 11) * (1.0 / 9007199254740992.0)) - 1.0));
    }
    const double limo = sqrt(6.0 / (double)(W + 1));
    for (int t = qpr::OFF_WO; t < qpr::OFF_BO; ++t)
        th[t] = (float)(limo * (2.0 * ((double)(qpr::splitmix(st) >> 11) * (1.0 / 9007199254740992.0)) - 1.0));
    if (cudaMemcpy(g->theta, th.data(), P * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(g->m, 0, P * sizeof(float)) != cudaSuccess || cudaMemset(g->v, 0, P * sizeof(float)) != cudaSuccess)
        return bail(gnn_fail(nullptr, QPR_E_CUDA, "parameter upload failed"));
    qpr::round_params_kernel<<<(P + 255) / 256, 256, 0, g->stream>>>(g->theta, g->fwd, P);
    if (cudaStreamSynchronize(g->stream) != cudaSuccess) return bail(gnn_fail(nullptr, QPR_E_CUDA, "init failed"));
    *out = g;
    return QPR_OK;
}

qpr_status qpr_gnn_get_params(qpr_gnn *g, float *host) {
    if (!g || !host) return QPR_E_ARG;
    cudaSetDevice(g->device);
    GCUDA(g, cudaMemcpy(host, g->theta, qpr::kParams * sizeof(float), cudaMemcpyDeviceToHost));
    return QPR_OK;
}

qpr_status qpr_gnn_set_params(qpr_gnn *g, const float *host) {
    if (!g || !host) return QPR_E_ARG;
    cudaSetDevice(g->device);
    GCUDA(g, cudaMemcpy(g->theta, host, qpr::kParams * sizeof(float), cudaMemcpyHostToDevice));
    qpr::round_params_kernel<<<(qpr::kParams + 255) / 256, 256, 0, g->stream>>>(g->theta, g->fwd, qpr::kParams);
    GCUDA(g, cudaMemset(g->m, 0, qpr::kParams * sizeof(float)));
    GCUDA(g, cudaMemset(g->v, 0, qpr::kParams * sizeof(float)));
    g->adam_t = 0;
    GCUDA(g, cudaStreamSynchronize(g->stream));
    return QPR_OK;
}

qpr_status qpr_gnn_predict(qpr_gnn *g, int64_t n, int64_t m, const int64_t *src, const int64_t *dst, const double *w,
                           double alpha, double omega, double *p_hat) {
    if (!g || !p_hat) return QPR_E_ARG;
    if (n < 2 || !(alpha >= 0.0 && alpha <= 1.0) || !(omega >= 0.0 && omega <= 1.0))
        return gnn_fail(g, QPR_E_ARG, "n < 2 or alpha/omega outside [0, 1]");
    cudaSetDevice(g->device);
    qpr::HostGraph hg;
    std::string e;
    qpr_status st = qpr::build_graph(n, m, src, dst, w, alpha, omega, hg, e);
    if (st != QPR_OK) return gnn_fail(g, st, e);
    qpr::GnnDev d;
    st = single_pass(g, hg, nullptr, false, &d);
    if (st != QPR_OK) return st;
    GCUDA(g, cudaMemcpyAsync(p_hat, d.p_hat, n * sizeof(double), cudaMemcpyDefault, g->stream));
    GCUDA(g, cudaStreamSynchronize(g->stream));
    GCUDA(g, cudaGetLastError());
    return QPR_OK;
}

qpr_status qpr_gnn_loss_grad(qpr_gnn *g, const qpr_gnn_sample *smp, double alpha, double *loss, float *grad) {
    if (!g || !smp || !smp->p) return QPR_E_ARG;
    cudaSetDevice(g->device);
    qpr::HostGraph hg;
    std::string e;
    qpr_status st = qpr::build_graph(smp->n, smp->m, smp->src, smp->dst, smp->w, alpha, smp->omega, hg, e);
    if (st != QPR_OK) return gnn_fail(g, st, e);
    qpr::GnnDev d;
    st = single_pass(g, hg, smp->p, true, &d);
    if (st != QPR_OK) return st;
    if (loss) GCUDA(g, cudaMemcpyAsync(loss, g->loss, sizeof(double), cudaMemcpyDeviceToHost, g->stream));
    if (grad) GCUDA(g, cudaMemcpyAsync(grad, g->grad, qpr::kParams * sizeof(float), cudaMemcpyDeviceToHost, g->stream));
    GCUDA(g, cudaStreamSynchronize(g->stream));
    GCUDA(g, cudaGetLastError());
    return QPR_OK;
}

qpr_status qpr_gnn_train(qpr_gnn *g, int64_t count, const qpr_gnn_sample *samples, double alpha, int32_t epochs,
                         int32_t batch, double lr, uint64_t seed, double *epoch_loss) {
    if (!g || count < 1 || !samples || epochs < 1 || batch < 1 || !(lr > 0.0)) return QPR_E_ARG;
    cudaSetDevice(g->device);
    std::vector<qpr::HostGraph> hg((size_t)count);
    for (int64_t i = 0; i < count; ++i) {
        if (!samples[i].p) return gnn_fail(g, QPR_E_ARG, "sample without target populations");
        std::string e;
        const qpr_status st = qpr::build_graph(samples[i].n, samples[i].m, samples[i].src, samples[i].dst,
                                               samples[i].w, alpha, samples[i].omega, hg[i], e, count > 4);
        if (st != QPR_OK) return gnn_fail(g, st, "sample " + std::to_string(i) + ": " + e);
    }
    // the graphs: all on the device, or a group at a time
    size_t total = 0;
    for (const qpr::HostGraph &h : hg) total += graph_bytes(h);
    const bool resident = total <= kResidentBytes;
    std::vector<qpr::GnnDev> graphs((size_t)count);
    std::vector<char> img;
    auto upload = [&](const std::vector<int64_t> &ids) -> qpr_status {
        std::vector<const qpr::HostGraph *> h;
        std::vector<const double *> p;
        std::vector<qpr::GnnDev *> d;
        for (int64_t i : ids) {
            h.push_back(&hg[i]);
            p.push_back(samples[i].p);
            d.push_back(&graphs[i]);
        }
        return upload_graphs(g, h, p, d, img);
    };
    for (int64_t i = 0; i < count;) {
        // a set that does not stay: its features come back once, part by part
        std::vector<int64_t> ids;
        size_t bytes = 0;
        for (; i < count && (ids.empty() || bytes + graph_bytes(hg[i]) <= kResidentBytes); ++i) {
            ids.push_back(i);
            bytes += graph_bytes(hg[i]);
        }
        const qpr_status st = upload(ids);
        if (st != QPR_OK) return st;
        if (resident) break;
        for (int64_t k : ids) {
            GCUDA(g, cudaMemcpyAsync(hg[k].x.data(), graphs[k].x, hg[k].x.size() * sizeof(float), cudaMemcpyDeviceToHost,
                                     g->stream));
            hg[k].device_pr = false;
        }
        GCUDA(g, cudaStreamSynchronize(g->stream));
    }
    {
        const qpr_status st = grow_desc(g, (size_t)count);
        if (st != QPR_OK) return st;
    }
    std::vector<int64_t> order((size_t)count);
    for (int64_t i = 0; i < count; ++i) order[i] = i;
    uint64_t rs = seed;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int ep = 0; ep < epochs; ++ep) {
        for (int64_t i = count - 1; i > 0; --i) std::swap(order[i], order[qpr::splitmix(rs) % (uint64_t)(i + 1)]);
        GCUDA(g, cudaMemsetAsync(g->loss, 0, sizeof(double), g->stream));
        for (int64_t b0 = 0; b0 < count; b0 += batch) {
            const int64_t b1i = std::min<int64_t>(count, b0 + batch);
            for (int64_t k = b0; k < b1i;) {
                std::vector<int64_t> ids;
                int maxn = 0;
                size_t bytes = 0;
                for (; k < b1i && (ids.empty() || bytes + ws_bytes(hg[order[k]].n) <= kGroupBytes); ++k) {
                    ids.push_back(order[k]);
                    bytes += ws_bytes(hg[order[k]].n);
                    maxn = std::max(maxn, hg[order[k]].n);
                }
                const bool init = (int64_t)ids.size() == k - b0;  // the batch's first group
                if (!resident) {
                    const qpr_status st = upload(ids);
                    if (st != QPR_OK) return st;
                }
                // an epoch uses each descriptor slot once and ends with a wait
                qpr::GnnDev *grp = g->desc + (k - (int64_t)ids.size()), *dev = nullptr;
                for (size_t q = 0; q < ids.size(); ++q) grp[q] = graphs[ids[q]];
                const qpr_status st = place_group(g, grp, ids.size(), &dev);
                if (st != QPR_OK) return st;
                enqueue_pass(g, dev, (int)ids.size(), maxn, true, init);
            }
            ++g->adam_t;
            const float c1 = 1.f - powf(b1, (float)g->adam_t), c2 = 1.f - powf(b2, (float)g->adam_t);
            qpr::adam_kernel<<<(qpr::kParams + 255) / 256, 256, 0, g->stream>>>(
                g->theta, g->fwd, g->grad, g->m, g->v, 1.f / (float)(b1i - b0), (float)lr, b1, b2, eps, c1, c2,
                qpr::kParams);
        }
        double l = 0.0;
        GCUDA(g, cudaMemcpyAsync(&l, g->loss, sizeof(double), cudaMemcpyDeviceToHost, g->stream));
        GCUDA(g, cudaStreamSynchronize(g->stream));
        GCUDA(g, cudaGetLastError());
        if (epoch_loss) epoch_loss[ep] = l / (double)count;
    }
    return QPR_OK;
}

}  // extern "C"
