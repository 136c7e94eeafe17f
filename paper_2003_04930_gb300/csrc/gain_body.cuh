// FP64 gain g = G p as a device function (single-problem and batched kernels).
#pragma once

#include <math.h>

#include "qpr_internal.cuh"

namespace qpr {
namespace gain64 {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The threads that work together: a whole CTA, or its warps from `FIRST` on
// (synchronised by barrier 1).
struct Cta {
    __device__ __forceinline__ int tid() const { return threadIdx.x; }
    __device__ __forceinline__ int size() const { return blockDim.x; }
    __device__ __forceinline__ void sync() const { __syncthreads(); }
};
template <int FIRST, int THREADS>
struct Warps {
    __device__ __forceinline__ int tid() const { return threadIdx.x - 32 * FIRST; }
    __device__ __forceinline__ int size() const { return THREADS; }
    __device__ __forceinline__ void sync() const { asm volatile("bar.sync 1, %0;\n" ::"n"(THREADS) : "memory"); }
};

// Fixed-order sum over the group, broadcast to every thread (1024 at most).
template <typename G = Cta>
__device__ __forceinline__ double block_sum(double v, double *red, G grp = G{}) {
    const int lane = threadIdx.x & 31, warp = grp.tid() >> 5;
    v = warp_sum(v);
    grp.sync();  // red may still be read by a previous call
    if (lane == 0) red[warp] = v;
    grp.sync();
    double s = 0.0;
    const int nw = (grp.size() + 31) >> 5;
    for (int q = 0; q < nw; ++q) s += red[q];
    return s;
}

// The stop decision of stage 2: the residual partials of stage 1 summed in
// index order into ||f(y_n)||_F of the normalised state. One group of threads.
template <typename G = Cta>
__device__ __forceinline__ void stop_decision(const Work &w, double *red, G grp = G{}) {
    Ctl *ctl = w.ctl;
    double s = 0.0;
    for (int i = grp.tid(); i < w.npairs; i += grp.size()) s += w.partials[i];
    s = block_sum(s, red, grp);
    if (grp.tid() == 0) {
        const double r = ctl->scale * sqrt(s);
        ctl->resid = r;
        ctl->resid_step = ctl->step;
        if (!isfinite(r)) {
            ctl->status = kCtlNonFinite;
            ctl->done = 1;
        } else if (r < ctl->tol) {
            ctl->status = kCtlConverged;
            ctl->done = 1;
        } else if (ctl->step >= ctl->max_steps) {
            ctl->status = kCtlMaxSteps;
            ctl->done = 1;
        }
    }
}

// out[i - base] = g_i for rows i = r0 + (warp of the group), + step, ... < r1,
// g = G p with G = alpha S + (1 - alpha) F (Eq. S2, Eq. S4), p_j = Y_jj
// (diag[j stride]):
//   (S p)_i = sum_{j with out-links} A_ij / outDeg(j) p_j  +  dangling part,
//   dangling part = (D - [i dangles] p_i) / (N - 1)  (F columns)  or  D / N,
//   (F p)_i = (P - p_i) / (N - 1),
// with P = sum_j p_j and D = sum over dangling j of p_j. With `publish` (one
// group of stage 1) it also sets 1 / Re tr(y), by which stage 4 normalises.
template <typename G = Cta>
__device__ __forceinline__ void gain_rows(const DevOps &ops, Ctl *ctl, const double *__restrict__ diag, size_t stride,
                                          int r0, int step, int r1, int base, double *out, bool publish, double *red,
                                          G grp = G{}) {
    const int n = ops.n;
    // independent of the sums below: the reciprocal, and the row sum of this
    // warp's first row, whose loads then fly with those of the diagonal
    const double inv_nm1 = __drcp_rn((double)(n - 1));
    const int lane = threadIdx.x & 31;
    const int first = r0 + (grp.tid() >> 5);
    auto row_part = [&](int i) {
        double s = 0.0;
        if (i < n) {
            for (int q = ops.s_ptr[i] + lane; q < ops.s_ptr[i + 1]; q += 32)
                s = __fma_rn(ops.s_val[q], diag[ops.s_col[q] * stride], s);
        }
        return s;
    };
    const double s0 = first < r1 ? row_part(first) : 0.0;
    double P = 0.0, D = 0.0;
    for (int j = grp.tid(); j < n; j += grp.size()) {
        const double pj = diag[j * stride];
        P += pj;
        if (ops.dang[j]) D += pj;
    }
    P = block_sum(P, red, grp);
    D = block_sum(D, red, grp);
    if (publish && grp.tid() == 0) {
        ctl->scale = 1.0 / P;
        ctl->trace = P;
        if (!(P > 0.0) || !isfinite(P)) {
            ctl->status = kCtlNonFinite;
            ctl->done = 1;
        }
    }
    for (int i = first; i < r1; i += step) {
        const double s = warp_sum(i == first ? s0 : row_part(i));
        if (lane == 0) {
            double gi = 0.0;
            if (i < n) {
                const double pi = diag[i * stride];
                const double dterm = (ops.dangling == QPR_DANGLING_F)
                                         ? __dmul_rn(__dsub_rn(D, ops.dang[i] ? pi : 0.0), inv_nm1)
                                         : __ddiv_rn(D, (double)n);
                gi = __fma_rn(ops.alpha, __dadd_rn(s, dterm),
                              __dmul_rn(__dmul_rn(__dsub_rn(1.0, ops.alpha), __dsub_rn(P, pi)), inv_nm1));
            }
            out[i - base] = gi;
        }
    }
}

// The gain of a stage into w.g by nblk groups of threads, this one blk; stage
// 1 publishes the scale, stage 2 takes the stop decision (group 0 both).
template <typename G = Cta>
__device__ __forceinline__ void gain_fp64_body(int stage, const DevOps &ops, const Work &w,
                                               const double *__restrict__ diag, size_t stride, int blk, int nblk,
                                               G grp = G{}) {
    __shared__ double red[32];
    if (stage == 2 && blk == 0) stop_decision(w, red, grp);
    const int wpb = grp.size() >> 5;
    gain_rows(ops, w.ctl, diag, stride, blk * wpb, nblk * wpb, ops.np, 0, w.g, stage == 1 && blk == 0, red, grp);
}

}  // namespace gain64
}  // namespace qpr
