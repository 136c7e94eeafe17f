// Fused FP64 epilogue shared by the RK4 stage kernels (dense digits, dense
// DMMA, sparse CSR).
//
// Input, in shared memory, for the tile pair (I, J), I <= J, of 32 x 32
// complex tiles: sX1 holds X = H Y restricted to rows I and columns J,
// sX2 the same for rows J and columns I (sX2 == sX1 when I == J), each as
// [32][ldx] doubles with
//     sX[a * ldx + b]      = (H Re Y)_ab,
//     sX[a * ldx + 32 + b] = -(H Im Y)_ab.
// With X = A + iB the Lindblad right-hand side (Eq. 1 / Eq. S7, with the
// jump operators L_ij = sqrt(G_ij)|i><j|) of entry (a, b) is
//     k_ab = (1-omega) [ (B_ab + B_ba) - i (A_ab - A_ba) ]
//            + omega [ delta_ab g_a - 1/2 (c_a + c_b) Y_ab ].
// f is linear, so the classical RK4 step (Supplementary Note 2) is the same
// polynomial in the nested form
//     y <- y + dt f(y + dt/2 f(y + dt/3 f(y + dt/4 f(y)))),
// which keeps no running sum: stages 1-3 write the next stage input
// y + c dt k (c = 1/4, 1/3, 1/2) and stage 4 the new y. The trace
// normalisation is linear too: the stages work on the unnormalised y and
// stage 4 multiplies by 1 / tr(y). Tile (I, J) is written directly and tile
// (J, I) as its conjugate transpose through shared memory, so every state
// stays exactly Hermitian.
//
// What bounds it: the FP64 pipe (two operations a clock and SM) and, in a
// small grid, the latency of its loads. So an element costs 10 FP64
// operations a stage (11 in the digit products; 15 to 17 with the running sum
// and a normalisation per stage, and two divisions per thread before), and all of a thread's
// operands are loaded together by EpiIn::load: at N = 500 (136 pairs) 18.6 us
// a launch before, 9.3 now (both with cold caches), 4.2 within a step.
#pragma once

#include "qpr_internal.cuh"

namespace qpr {

constexpr int kEpiTS = 32;

__device__ __forceinline__ double epi_warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The operands of this thread's elements e = tid + NT i of the 32 x 32 tile
// (I, J): the stage input and, where it differs, y; the decay rates of the
// rows and of the column; the step's scalars. Read through L2: a dependent
// launch may load them while the kernel before it still runs, when they were
// written before that one began.
template <int STAGE, int NT>
struct EpiIn {
    static constexpr int E = kEpiTS * kEpiTS / NT;
    double ir[E], ii[E], yr[E], yi[E], ca[E], cb, dt, scale;

    // c: ops.c, or what the product's form makes of it
    __device__ __forceinline__ void load(const DevOps &ops, const Work &w, int I, int J, const double *c) {
        const size_t plane = (size_t)ops.np * ops.np;
        const double *yin = (STAGE <= 1) ? w.y : (STAGE == 3 ? w.yb : w.ya);
        const int b = threadIdx.x & 31;
        cb = c[J * kEpiTS + b];
        dt = __ldcg(&w.ctl->dt);
        scale = (STAGE == 4) ? __ldcg(&w.ctl->scale) : 1.0;
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const int ga = I * kEpiTS + (threadIdx.x >> 5) + i * (NT / 32);
            const size_t off = (size_t)ga * ops.np + J * kEpiTS + b;
            ir[i] = __ldcg(yin + off);
            ii[i] = __ldcg(yin + plane + off);
            yr[i] = (STAGE >= 2) ? __ldcg(w.y + off) : ir[i];
            yi[i] = (STAGE >= 2) ? __ldcg(w.y + plane + off) : ii[i];
            ca[i] = c[ga];
        }
    }
};

// What differs between the products: the decay rate omega / 2 (c_a + c_b) from
// what EpiIn holds for row and column (the digit products' epilogue holds
// omega / 2 c, one operation less), and what the product left out of A_ab - A_ba of
// element i (the digit products: the diagonal of the stage input).
struct WholeProduct {
    __device__ __forceinline__ double rate(double hom, double ca, double cb) const {
        return __dmul_rn(hom, __dadd_rn(ca, cb));
    }
    __device__ __forceinline__ double difference(int, double d) const { return d; }
};

// Must be called by all NT threads of the CTA after the X tiles are complete
// and visible (__syncthreads()). Off the diagonal sX1 is overwritten with the
// outputs, each by the one thread that reads that place.
// g: the gain of rows I, read on diagonal pairs. pidx: slot of this tile
// pair's residual partial; first: the tile pair that advances the step counter
// at stage 4. form: WholeProduct or its like.
template <int STAGE, int NT, typename P = WholeProduct>
__device__ __forceinline__ void stage_epilogue(const DevOps &ops, const Work &w, int I, int J, bool diag,
                                               const EpiIn<STAGE, NT> &in, double *sX1, const double *sX2, int ldx,
                                               const double *g, double *red, int pidx, bool first,
                                               const P &form = P{}) {
    constexpr int TS = kEpiTS, E = EpiIn<STAGE, NT>::E;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int np = ops.np;
    const size_t plane = (size_t)np * np;
    const double *X2 = diag ? sX1 : sX2;
    const double om = ops.omega, cm = 1.0 - om;
    const double dt = in.dt, scale = in.scale;
    const double cst = (STAGE == 1) ? 0.25 * dt : STAGE == 2 ? __dmul_rn(dt, 1.0 / 3.0) : STAGE == 3 ? 0.5 * dt : dt;
    double *dst = (STAGE == 0) ? w.z : STAGE == 4 ? w.y : (STAGE == 2 ? w.yb : w.ya);
    double nrm = 0.0;

    // Every operation below is an explicit round-to-nearest intrinsic, so the
    // result does not depend on how a compiler contracts it in the kernel that
    // inlines this function (single-problem and batched kernels agree bitwise).
    const double hom = 0.5 * om;
    const int b = lane, gb = J * TS + b;
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const int a = warp + i * (NT / 32), ga = I * TS + a;
        const size_t off = (size_t)ga * np + gb;
        const double Aab = sX1[a * ldx + b], nBab = sX1[a * ldx + TS + b];
        const double Aba = X2[b * ldx + a], nBba = X2[b * ldx + TS + a];
        const double omhc = form.rate(hom, in.ca[i], in.cb);  // the same for (b, a)
        double kr = __fma_rn(-omhc, in.ir[i], __dmul_rn(-cm, __dadd_rn(nBab, nBba)));
        const double ki = __fma_rn(-omhc, in.ii[i], __dmul_rn(-cm, form.difference(i, __dsub_rn(Aab, Aba))));
        if (ga == gb) kr = __fma_rn(om, g[a], kr);
        if (STAGE <= 1) nrm = __fma_rn(kr, kr, __fma_rn(ki, ki, nrm));
        double o0 = kr, o1 = ki;
        if (STAGE >= 1) {
            o0 = __fma_rn(cst, kr, in.yr[i]);
            o1 = __fma_rn(cst, ki, in.yi[i]);
        }
        if (STAGE == 4) {
            o0 = __dmul_rn(scale, o0);
            o1 = __dmul_rn(scale, o1);
        }
        dst[off] = o0;
        dst[plane + off] = o1;
        if (!diag) {
            sX1[a * ldx + b] = o0;
            sX1[a * ldx + TS + b] = o1;
        }
    }

    if (STAGE <= 1) {
        nrm = epi_warp_sum(nrm);
        if (lane == 0) red[warp] = nrm;
        __syncthreads();
        if (tid == 0) {
            double s = 0.0;
            for (int q = 0; q < NT / 32; ++q) s += red[q];
            w.partials[pidx] = diag ? s : 2.0 * s;
        }
    }

    if (!diag) {
        __syncthreads();
        // tile (J, I) = conjugate transpose of tile (I, J)
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const int r = warp + i * (NT / 32);
            const size_t off = (size_t)(J * TS + r) * np + I * TS + lane;
            dst[off] = sX1[lane * ldx + r];
            dst[plane + off] = -sX1[lane * ldx + TS + r];
        }
    }

    if (STAGE == 4 && first && tid == 0) w.ctl->step += 1;
}

}  // namespace qpr
