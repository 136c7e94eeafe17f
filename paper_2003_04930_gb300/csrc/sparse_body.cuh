// FP64 sparse stage: one tile pair as a device function (shared by the
// single-problem kernel and the batched kernels).
//
// What bounds it: the FP64 pipe, one warp instruction per scheduler in 40 ns.
// At N = 922 (16 nonzeros a row) the products are 856,000 warp instructions
// and the epilogue 139,000: 65 us a stage if every scheduler always had one
// to issue. So the work is spread evenly: rows of more than kCoop nonzeros
// (hubs) are shared by all warps of the CTA, the others are handed to the
// next free warp, and a row's entries are read 32 at a time, one per lane, so
// that a batch of four nonzeros waits for one L2 round trip, not two. The
// gain of a diagonal tile's rows is formed in its own CTA, which has half
// the products of the others (a launch of its own took 10 us a stage).
// Measured at N = 922: 162 us a stage before, 97 now (N = 1500: 390 and 200).
// The line at 96 is flat from 48 to 96 and 6% slower at 192 (N = 922).
#pragma once

#include "gain_body.cuh"
#include "qpr_internal.cuh"
#include "stage_epilogue.cuh"

namespace qpr {
namespace sparse64 {

constexpr int TS = kEpiTS;
constexpr int NTHREADS = 256;
constexpr int NWARPS = NTHREADS / 32;
constexpr int LDX = 2 * TS + 1;
constexpr int kCoop = 96;  // longer rows are shared by the CTA's warps
constexpr int SMEM_BYTES = (2 * TS * LDX + NWARPS * 2 * TS) * (int)sizeof(double);

// Entries [q0, q1) of a row of H times 32 columns of Y (yre, yim: this lane's
// column), added to (xr, xi) in entry order: explicit fused multiply-adds,
// the same rounding in every kernel that inlines this function.
__device__ __forceinline__ void row_product(const DevOps &ops, const double *__restrict__ yre,
                                            const double *__restrict__ yim, int q0, int q1, double &xr, double &xi) {
    const int lane = threadIdx.x & 31;
    const size_t np = ops.np;
    for (int qb = q0; qb < q1; qb += 32) {
        const int m = min(32, q1 - qb);
        int k = 0;
        double h = 0.0;
        if (lane < m) {
            k = ops.h_col[qb + lane];
            h = ops.h_val[qb + lane];
        }
        int e = 0;
        for (; e + 4 <= m; e += 4) {
            double r[4], i[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const size_t o = __shfl_sync(0xffffffffu, k, e + u) * np;
                r[u] = yre[o];
                i[u] = yim[o];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const double hu = __shfl_sync(0xffffffffu, h, e + u);
                xr = __fma_rn(hu, r[u], xr);
                xi = __fma_rn(hu, i[u], xi);
            }
        }
        for (; e < m; ++e) {
            const size_t o = __shfl_sync(0xffffffffu, k, e) * np;
            const double hu = __shfl_sync(0xffffffffu, h, e);
            xr = __fma_rn(hu, yre[o], xr);
            xi = __fma_rn(hu, yim[o], xi);
        }
    }
}

// sX1 = rows I of H times columns J of Y, sX2 = rows J times columns I (off
// the diagonal), each [TS][LDX]; part: NWARPS x 2 TS doubles. Ends with a
// barrier.
__device__ __forceinline__ void spmm_pair(const DevOps &ops, const double *__restrict__ yin, size_t plane, int I, int J,
                                          bool diag, double *sX1, double *sX2, double *part) {
    __shared__ int s_ptr[2][TS + 1];
    __shared__ int s_next;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = ops.n, rows = diag ? TS : 2 * TS;
    if (threadIdx.x < 2 * (TS + 1)) {
        const int t = threadIdx.x / (TS + 1), a = threadIdx.x - t * (TS + 1);
        s_ptr[t][a] = ops.h_ptr[min(n, (t ? J : I) * TS + a)];
    }
    if (threadIdx.x == 0) s_next = 0;
    __syncthreads();
    // item i: row i % TS of tile I (i < TS) or J
    for (int i = 0; i < rows; ++i) {
        const int t = i >= TS, a = i - t * TS;
        const int q0 = s_ptr[t][a], len = s_ptr[t][a + 1] - q0;
        if (len <= kCoop) continue;
        const double *y = yin + (t ? I : J) * TS + lane;
        double xr = 0.0, xi = 0.0;
        row_product(ops, y, y + plane, q0 + warp * len / NWARPS, q0 + (warp + 1) * len / NWARPS, xr, xi);
        part[warp * 2 * TS + lane] = xr;
        part[warp * 2 * TS + TS + lane] = xi;
        __syncthreads();
        if (threadIdx.x < 2 * TS) {
            double s = part[threadIdx.x];
            for (int q = 1; q < NWARPS; ++q) s = __dadd_rn(s, part[q * 2 * TS + threadIdx.x]);
            (t ? sX2 : sX1)[a * LDX + threadIdx.x] = threadIdx.x < TS ? s : -s;
        }
        __syncthreads();
    }
    for (;;) {
        int i = 0;
        if (lane == 0) i = atomicAdd(&s_next, 1);
        i = __shfl_sync(0xffffffffu, i, 0);
        if (i >= rows) break;
        const int t = i >= TS, a = i - t * TS;
        const int q0 = s_ptr[t][a], q1 = s_ptr[t][a + 1];
        if (q1 - q0 > kCoop) continue;
        const double *y = yin + (t ? I : J) * TS + lane;
        double xr = 0.0, xi = 0.0;
        row_product(ops, y, y + plane, q0, q1, xr, xi);
        double *sX = (t ? sX2 : sX1) + a * LDX;
        sX[lane] = xr;
        sX[TS + lane] = -xi;
    }
    __syncthreads();
}

// One tile pair (I, J) of stage STAGE; smem: SMEM_BYTES of dynamic shared
// memory. The pair (0, 0) publishes the scale at stage 1 and takes the stop
// decision at stage 2 (whose outputs are scratch if the run stops there).
// Ends with a barrier so that the caller may reuse shared memory.
template <int STAGE>
__device__ __forceinline__ void tile(const DevOps &ops, const Work &w, int I, int J, int pidx, bool first,
                                     double *smem) {
    __shared__ double red[32];
    __shared__ double sg[TS];
    const bool diag = (I == J);
    const size_t plane = (size_t)ops.np * ops.np;
    const double *__restrict__ yin = (STAGE <= 1) ? w.y : (STAGE == 3 ? w.yb : w.ya);
    double *sX1 = smem;
    double *sX2 = smem + TS * LDX;
    if (STAGE == 2 && diag && I == 0) gain64::stop_decision(w, red);
    if (diag)
        gain64::gain_rows(ops, w.ctl, yin, (size_t)ops.np + 1, I * TS, NWARPS, I * TS + TS, I * TS, sg,
                          STAGE == 1 && I == 0, red);
    spmm_pair(ops, yin, plane, I, J, diag, sX1, sX2, smem + 2 * TS * LDX);
    EpiIn<STAGE, NTHREADS> in;
    in.load(ops, w, I, J, ops.c);  // after the product: its registers are free (725 -> 615 us a step at N = 922)
    stage_epilogue<STAGE, NTHREADS>(ops, w, I, J, diag, in, sX1, sX2, LDX, sg, red, pidx, first);
    __syncthreads();
}

}  // namespace sparse64
}  // namespace qpr
