// FP64 dense RK4 stage with the product on the 5th-generation tensor cores:
// X = H Y from exact integer digit products (the splitting of Ozaki, Ogita,
// Oishi and Rump, "Error-free transformations of matrix multiplication",
// 2012, with integer digits).
//
// Why: FP64 runs at 1.04 TFLOP/s on this part, FP16 with FP32 accumulation at
// about 1900. The FP64 tensor instruction (stage_fp64.cu) took 616 us per
// stage at N = 500 (4.2 ms at N = 922), one 32 x 32 tile pair per CTA; this
// form takes 26 us at N = 500 with unit weights and 362 us at N = 922 with
// lognormal ones. Here every entry off the diagonal is written as
//     Y_jk = 2^(ec_j) sum_s y_s(j, k) 2^(-b s),   s < S,  |y_s| <= 2^(b-1),
// with integers y_s (exact in FP16) and ec_j from the largest entry of row j
// off the diagonal, so S b >= 64 bits of every column of Y enter the product,
// and H likewise (one digit when its entries are small multiples of one power
// of two, as with unit weights; else S digits of its own row). The products of
// digits i and j with i + j = d share a weight, and all of them are summed in
// one FP32 accumulator that stays an integer below 2^24: exact in any order.
//
// What is left out: the digits after the S-th and, where H has several, the
// pairs with i + j >= S, together at most
//     5 S 2^(-S b) nnz(row i of H) max|H_i| max|Y_j|
// of X_ij, max|Y_j| the largest entry of column j off the diagonal; then one
// rounding (and at b = 10 one of the low half's 54 bits). The bound is relative
// to these largest entries: an entry of Y further below its column's largest
// than S b - 53 bits (11 to 19) enters with fewer than FP64's 53 bits. The
// diagonal, which is what towers over a column in a state with small
// coherences, therefore stays out of the product and is added in FP64 by the
// epilogue as H_ab (Y_bb - Y_aa) (DiagonalTerm): with it in the product,
// entries of pairs that are not linked were off by up to 1e-13 of their terms
// with coherences of 1e-5 / N and 1e-10 with 1e-8 / N, now 1e-16 (CPU model, N =
// 60, lognormal weights; FMA chains 1e-16).
//
// Kernels of a stage: split_kernel (digits of the stage input, a row per
// CTA), digits_gemm_kernel (one 128 x 32 tile of [H Re Y | -H Im Y] per CTA;
// the warps that wait for the product form the gain and take the stop
// decision, gain64::gain_fp64_body) and digits_epi_kernel (the fused Lindblad / RK4 epilogue
// of stage_epilogue.cuh per 32 x 32 tile pair). At N = 500 a stage is latency
// from end to end, so they are launched with programmatic dependent launch
// and do what they can before they wait: the product kernel allocates TMEM
// and loads H, the epilogue loads its operands but X and the gain. (The
// epilogue starts once every CTA of the product has passed its own wait, so
// the split kernel before that and everything older is complete.)
//
// The tile: 128 rows (the MMA's M) by 32 columns of one plane, all S digits
// of these columns stacked as the MMA's N, so the accumulators of all weights
// fill S x 32 TMEM columns and one instruction multiplies a digit plane of H
// with every digit it pairs with (N = 192 of 256 with one digit of H and
// S = 6). 32 columns because the small problems need the CTAs: N = 500 gives
// 128 of them.
#include <cuda.h>
#include <cuda_fp16.h>
#include <math.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "gain_body.cuh"
#include "qpr_internal.cuh"
#include "stage_epilogue.cuh"
#include "tma_util.cuh"

namespace qpr {
namespace {

constexpr int TM = 128;                 // rows of a tile
constexpr int TN = 32;                  // columns of a tile (one plane)
constexpr int BK = 64;                  // FP16 k per block: one 128-byte swizzle row
constexpr int A_BYTES = TM * BK * 2;    // 16 KB per digit plane of H
constexpr int B_ROW = TN * BK * 2;      // 4 KB per digit of Y
constexpr int kMaxDigits = 13;
constexpr int kMaxRing = 4;
constexpr int GT = 256;                 // threads of the GEMM kernel
constexpr int LDT = TN + 1;             // staged output tile row
constexpr int kNanExp = 1 << 20;        // marks a row of Y that is not finite

using tma::load_3d;
using tma::load_4d;
using tma::mbar_expect_tx;
using tma::mbar_init;
using tma::mbar_wait;
using tma::smem_u32;

// The digits of x in units of 2^e (the unit of the last digit): x / 2^e
// rounded to an integer V, |V| < 2^(b S - 1), as S base-2^b digits in
// [-2^(b-1), 2^(b-1)], the first one the most significant. Integer
// instructions only (the FP64 pipe is the scarce one).
__host__ __device__ __forceinline__ void digits_of(double x, int e, int S, int b, int16_t *d) {
    long long bits;
#ifdef __CUDA_ARCH__
    bits = __double_as_longlong(x);
#else
    memcpy(&bits, &x, 8);
#endif
    const int ex = (int)((bits >> 52) & 0x7ff);
    unsigned long long m = (unsigned long long)bits & 0xfffffffffffffull;
    if (ex) m |= 1ull << 52;
    const int sh = (ex ? ex : 1) - 1075 - e;
    __int128 v = 0;
    if (sh >= 0) v = (__int128)m << (sh > 74 ? 74 : sh);
    else if (sh > -64) v = (__int128)((m + (1ull << (-sh - 1))) >> -sh);
    if (bits < 0) v = -v;
    // add half a base to every digit but the first: each is then a field of
    // b bits, its half taken off again
    const int half = 1 << (b - 1), mask = (1 << b) - 1;
    for (int s = S - 1; s > 0; --s) {
        v += half;
        d[s] = (int16_t)(((int)v & mask) - half);
        v >>= b;
    }
    d[0] = (int16_t)(int)v;
}

// exponent of the least power of two above |x| (finite, from the high word)
__host__ __device__ __forceinline__ int exp_above(unsigned hi) { return (int)((hi >> 20) & 0x7ff) - 1022; }

// A row of Y per CTA, two warps to a plane: each plane's largest exponent,
// then the digits. Bound by the latency of its loads and by integer
// instructions: the loads are issued four at a time and kept for the digits
// where a lane has no more of them (N <= 512); one warp per row and plane took
// 8.4 us at N = 500, this 5.
template <int S, int B>
__global__ void __launch_bounds__(128) split_kernel(DevOps ops, Ctl *ctl, const double *__restrict__ y, DigitWork dw) {
    __shared__ int s_done;
    __shared__ unsigned s_top[4];
    tma::grid_dependency_wait();
    tma::launch_dependents();
    if (threadIdx.x == 0) s_done = *(volatile int *)&ctl->done;
    __syncthreads();
    if (s_done) return;
    constexpr int U = 4;  // loads in flight
    const int np = ops.np, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = blockIdx.x, pl = warp >> 1;
    const size_t plane = (size_t)np * np;
    const double2 *src = reinterpret_cast<const double2 *>(y + pl * plane + (size_t)row * np);
    const int k0 = (warp & 1) * 32 + lane, nk = np / 2;
    double2 v[U];
    // the diagonal entry stays outside the product (DiagonalTerm); the gain and
    // the epilogue read it from a vector
    const double yd = threadIdx.x == 0 ? y[(size_t)row * (np + 1)] : 0.0;
    auto load = [&](int k) {
        double2 r = k < nk ? src[k] : make_double2(0.0, 0.0);
        if (k == row >> 1) (row & 1 ? r.y : r.x) = 0.0;
        return r;
    };
    unsigned top = 0;
    for (int k = k0; k < nk; k += 64 * U) {
#pragma unroll
        for (int i = 0; i < U; ++i) v[i] = load(k + 64 * i);
#pragma unroll
        for (int i = 0; i < U; ++i)
            top = max(top, max((unsigned)__double2hiint(v[i].x) & 0x7fffffffu, (unsigned)__double2hiint(v[i].y) & 0x7fffffffu));
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) s_top[warp] = top;
    __syncthreads();
    top = max(s_top[2 * pl], s_top[2 * pl + 1]);
    const int ea = exp_above(top);
    const int e0 = ea - (B - 1);  // unit of the first digit
    if (threadIdx.x == 0) dw.diag[row] = yd;
    if ((warp & 1) == 0 && lane == 0) dw.ecol[pl * np + row] = (top >= 0x7ff00000u) ? kNanExp : e0;
    __half2 *dst = reinterpret_cast<__half2 *>(dw.yd) + (pl * plane + (size_t)row * np) / 2;
    const int eu = e0 - B * (S - 1);
    for (int k = k0; k < nk; k += 64 * U) {
        if (nk > 64 * U) {
#pragma unroll
            for (int i = 0; i < U; ++i) v[i] = load(k + 64 * i);
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            if (k + 64 * i >= nk) break;
            int16_t d0[S], d1[S];
            digits_of(v[i].x, eu, S, B, d0);
            digits_of(v[i].y, eu, S, B, d1);
#pragma unroll
            for (int s = 0; s < S; ++s)
                dst[s * plane + k + 64 * i] = __halves2half2(__short2half_rn(d0[s]), __short2half_rn(d1[s]));
        }
    }
}

// Digits of the entries of H into the zeroed planes hd [sh][np][np], and with
// several digits the entries themselves into the zeroed plane hf; omega / 2 c
// into hc.
__global__ void split_h_kernel(DevOps ops, int b, int sh, const int *__restrict__ erow, __half *hd, double *hf,
                               double *hc) {
    const size_t plane = (size_t)ops.np * ops.np;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ops.np; i += gridDim.x * blockDim.x)
        hc[i] = __dmul_rn(0.5 * ops.omega, ops.c[i]);
    for (int i = blockIdx.x; i < ops.n; i += gridDim.x)
        for (int q = ops.h_ptr[i] + threadIdx.x; q < ops.h_ptr[i + 1]; q += blockDim.x) {
            int16_t d[kMaxDigits];
            digits_of(ops.h_val[q], erow[i] - b * (sh - 1), sh, b, d);
            if (sh > 1) hf[(size_t)i * ops.np + ops.h_col[q]] = ops.h_val[q];
            for (int s = 0; s < sh; ++s) hd[s * plane + (size_t)i * ops.np + ops.h_col[q]] = __short2half_rn(d[s]);
        }
}

// Shared-memory matrix descriptor of a K-major operand in the 128-byte
// swizzled layout that TMA writes (8 rows x 128 B atoms, 1024 B apart).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)((1024 >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// kind::f16 with FP16 A and B (K-major), FP32 D, M = 128.
__device__ __forceinline__ uint32_t idesc_f16(int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}
__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(bar))
                 : "memory");
}
// Eight columns of this warp's TMEM lanes; tmem_wait makes them valid (its
// operands keep every use behind it).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
template <int S>
__device__ __forceinline__ void tmem_wait(uint32_t (&v)[S][8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int d = 0; d < S; ++d)
        asm volatile("" : "+r"(v[d][0]), "+r"(v[d][1]), "+r"(v[d][2]), "+r"(v[d][3]), "+r"(v[d][4]), "+r"(v[d][5]),
                          "+r"(v[d][6]), "+r"(v[d][7]));
}
// v 2^e, e added to the exponent where that stays a normal number.
__device__ __forceinline__ double scaled(double v, int e) {
    const int hi = __double2hiint(v), ex = ((hi >> 20) & 0x7ff) + e;
    if (v == 0.0) return v;
    if (ex > 0 && ex < 0x7ff) return __hiloint2double(hi + e * (1 << 20), __double2loint(v));
    return scalbn(v, e);
}

template <int S, int B>
__global__ void __launch_bounds__(GT) digits_gemm_kernel(const __grid_constant__ CUtensorMap tmH,
                                                         const __grid_constant__ CUtensorMap tmY, DevOps ops, Work w,
                                                         DigitWork dw, int stage) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t fullA[kMaxRing], emptyA[kMaxRing], fullB[kMaxRing], emptyB[kMaxRing], accum_bar;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int s_done, s_fail;
    Ctl *ctl = w.ctl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int np = ops.np, sh = dw.sh, ra = dw.ring_a, rb = dw.ring_b;
    const int tiles_m = (np + TM - 1) / TM;
    const int u = blockIdx.x;
    const int mt = u % tiles_m, ct = u / tiles_m;  // column tile: plane, then columns
    const int pl = ct / (np / TN), j0 = (ct - pl * (np / TN)) * TN;
    const int nkb = (np + BK - 1) / BK;
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *ringA = smem, *ringB = smem + ra * A_BYTES;
    const uint32_t tmem_cols = dw.tmem_cols;
    if (u >= tiles_m * (2 * np / TN)) {  // a CTA without a tile: a small problem's gain has more rows than its tiles' warps
        tma::grid_dependency_wait();
        tma::launch_dependents();
        if (warp >= 2) gain64::gain_fp64_body(stage, ops, w, dw.diag, 1, u, dw.gain_ctas, gain64::Warps<2, GT - 64>{});
        return;
    }

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_base_sh)),
                     "r"(tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    if (tid == 32) {
        for (int s = 0; s < kMaxRing; ++s) {
            mbar_init(&fullA[s], 1);
            mbar_init(&emptyA[s], 1);
            mbar_init(&fullB[s], 1);
            mbar_init(&emptyB[s], 1);
        }
        mbar_init(&accum_bar, 1);
        tma::mbar_init_fence();
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_base_sh;
    // the first digit planes of H do not depend on the kernel before
    const int ahead = min(ra, nkb * sh);
    auto load_h = [&](int ia) {
        const int sa = ia % ra;
        mbar_expect_tx(&fullA[sa], (uint32_t)A_BYTES);
        load_3d(ringA + sa * A_BYTES, &tmH, &fullA[sa], (ia / sh) * BK, mt * TM, ia % sh);
    };
    if (tid == 0)
        for (int ia = 0; ia < ahead; ++ia) load_h(ia);
    tma::grid_dependency_wait();
    tma::launch_dependents();
    if (tid == 0) {
        s_done = *(volatile int *)&ctl->done;
        s_fail = 0;
        if (s_done)  // nothing to do: let the loads land before the CTA ends
            for (int ia = 0; ia < ahead; ++ia) mbar_wait(&fullA[ia], 0);
    }
    __syncthreads();
    const bool work = !s_done;

    if (!work) {
    } else if (warp == 0 && lane == 0) {
        // producer: per k block the S digits of 32 rows of Y, then each digit plane of H
        int ia = 0;
        bool ok = true;
        for (int kb = 0; kb < nkb && ok; ++kb) {
            const int sb = kb % rb;
            if (kb >= rb) ok = mbar_wait(&emptyB[sb], ((kb / rb) - 1) & 1);
            if (!ok) break;
            mbar_expect_tx(&fullB[sb], (uint32_t)(S * B_ROW));
            load_4d(ringB + (size_t)sb * S * B_ROW, &tmY, &fullB[sb], kb * BK, j0, pl, 0);
            for (int i = 0; i < sh && ok; ++i, ++ia) {
                if (ia < ahead) continue;
                ok = mbar_wait(&emptyA[ia % ra], ((ia / ra) - 1) & 1);
                if (!ok) break;
                load_h(ia);
            }
        }
        if (!ok) atomicExch(&s_fail, 1);
    } else if (warp == 1 && lane == 0) {
        int ia = 0;
        bool ok = true;
        for (int kb = 0; kb < nkb && ok; ++kb) {
            const int sb = kb % rb;
            ok = mbar_wait(&fullB[sb], (kb / rb) & 1);
            for (int i = 0; i < sh && ok; ++i, ++ia) {
                const int sa = ia % ra;
                ok = mbar_wait(&fullA[sa], (ia / ra) & 1);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint64_t dA = sw128_desc(smem_u32(ringA + sa * A_BYTES));
                // digit i of H with digits 0 .. S - 1 - i of Y: weights i .. S - 1, at most 8 digits per instruction
                for (int j = 0; j < S - i; j += 8) {
                    const int nd = min(8, S - i - j);
                    const uint64_t dB = sw128_desc(smem_u32(ringB + ((size_t)sb * S + j) * B_ROW));
                    const uint32_t d = tmem + (uint32_t)((i + j) * TN), id = idesc_f16(nd * TN);
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
                        umma_f16(d, dA + (uint64_t)(kk * 2), dB + (uint64_t)(kk * 2), id, (kb | i | kk) ? 1u : 0u);
                }
                umma_commit(&emptyA[sa]);
            }
            umma_commit(&emptyB[sb]);
        }
        if (!ok) atomicExch(&s_fail, 1);
        umma_commit(&accum_bar);
    } else if (warp >= 2 && u < dw.gain_ctas) {
        gain64::gain_fp64_body(stage, ops, w, dw.diag, 1, u, dw.gain_ctas, gain64::Warps<2, GT - 64>{});
    }
    __syncwarp();
    const bool ok_acc = !work || mbar_wait(&accum_bar, 0);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (!work) {
    } else if (!ok_acc || s_fail) {
        if (tid == 0) atomicExch(&ctl->err_timeout, 1);
    } else {
        // Lane = row: the sums of the weights as one integer hi 2^low + lo,
        // then one FP64 value. hi (51 bits at most) becomes FP64 by writing
        // it into the low bits of 1.5 2^52, and lo, where it fits, into those
        // of 1.5 2^(52 - low): the difference of the first and both constants
        // is exact, the addition of the second rounds once. Two FP64
        // operations an element (the integer pipe does the rest); the scale
        // is added to the exponent. The pipeline buffers are free.
        double *sT = reinterpret_cast<double *>(smem);
        const int q = warp & 3, cb = (warp >> 2) * (TN / 2);  // rows of the warp (its TMEM lanes), its columns
        const int row = mt * TM + q * 32 + lane;
        const int er = row < ops.n ? dw.erow[row] : 0;
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        constexpr int nhi = S < 26 / B + 1 ? S : 26 / B + 1, low = B * (S - nhi);
        constexpr bool fits = 24 + B * (S - nhi - 1) <= 50;  // B = 12, 11, 8
        constexpr long long mhi = 0x4338000000000000ll, mlo = mhi - ((long long)low << 52);
        const double magic = 6755399441055744.0;  // 1.5 2^52
        const double both = magic + (fits ? __longlong_as_double(mlo) : 0.0);
        const double wlo = __longlong_as_double((long long)(1023 - low) << 52);  // 2^-low
        const int eu = er - B * (nhi - 1);  // the unit of hi's last digit
#pragma unroll 1
        for (int c0 = cb; c0 < cb + TN / 2; c0 += 8) {
            uint32_t v[S][8];
#pragma unroll
            for (int d = 0; d < S; ++d) tmem_ld8(tmem + lane_off + (uint32_t)(d * TN + c0), v[d]);
            int ec[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) ec[c] = dw.ecol[pl * np + j0 + c0 + c];
            tmem_wait(v);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                long long hi = 0, lo = 0;
#pragma unroll
                for (int d = 0; d < nhi; ++d) hi = hi * (1ll << B) + __float2int_rn(__uint_as_float(v[d][c]));
#pragma unroll
                for (int d = nhi; d < S; ++d) lo = lo * (1ll << B) + __float2int_rn(__uint_as_float(v[d][c]));
                const double h = __dsub_rn(__longlong_as_double(mhi + hi), both);
                const double x = fits ? __dadd_rn(h, __longlong_as_double(mlo + lo)) : __fma_rn((double)lo, wlo, h);
                sT[(q * 32 + lane) * LDT + c0 + c] =
                    (ec[c] == kNanExp) ? __longlong_as_double(0x7ff8000000000000ll) : scaled(x, eu + ec[c]);
            }
        }
        __syncwarp();
        // two rows of the warp's 16 columns per store
        const size_t plane = (size_t)np * np;
#pragma unroll 4
        for (int r = lane >> 4; r < 32; r += 2) {
            const int gr = mt * TM + q * 32 + r, c = cb + (lane & 15);
            if (gr < np) dw.x[pl * plane + (size_t)gr * np + j0 + c] = sT[(q * 32 + r) * LDT + c];
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(tmem_cols));
    }
}

constexpr int LDX = 2 * kEpiTS + 1;
constexpr int EPI_BYTES = 2 * kEpiTS * LDX * (int)sizeof(double);
// 512 threads, two elements each: a stage takes 20.3, 26.2 and 39.2 us at N =
// 100, 500 and 600 (unit weights), with 256 20.8, 26.0 and 44.9; from N = 1500
// on it makes no difference (183 and 185 us).
constexpr int ET = 512;

// k 2^t from its digit k != 0, by integer instructions (exact); 0 from 0.
__device__ __forceinline__ double from_digit(__half k, int t) {
    const unsigned f = __float_as_uint(__half2float(k));
    if ((f << 1) == 0) return 0.0;
    const unsigned hi = ((f & 0x7fffffffu) >> 3) + ((unsigned)(896 + t) << 20);  // the exponent rebiased, plus t
    return __hiloint2double((int)((f & 0x80000000u) | hi), (int)(f << 29));
}

// The diagonal's part of A_ab - A_ba, which the product leaves out: H_ab (Y_bb -
// Y_aa). H_ab in registers, from its one digit (ONE: no FP64 plane of H is
// kept) or from the plane d.h; the diagonal's entries of rows I and columns J
// in shared memory (in registers too a stage took 0.3 us longer at N = 500).
template <bool ONE>
struct DiagonalTerm {
    static constexpr int E = EpiIn<1, ET>::E;
    typename std::conditional<ONE, __half, double>::type h[E];
    const double *sd;  // Y_aa of the 32 rows, then Y_bb of the 32 columns
    int t;

    __device__ __forceinline__ void load(const DevOps &ops, const DigitWork &d, int I, int J, double *shared) {
        t = d.unit;
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const int ga = I * kEpiTS + (threadIdx.x >> 5) + i * (ET / 32);
            const size_t o = (size_t)ga * ops.np + J * kEpiTS + (threadIdx.x & 31);
            if constexpr (ONE) h[i] = __ldcg(reinterpret_cast<const __half *>(d.hd) + o);
            else h[i] = __ldcg(d.h + o);
        }
        if (threadIdx.x < 2 * kEpiTS)
            shared[threadIdx.x] = __ldcg(d.diag + (threadIdx.x < kEpiTS ? I : J) * kEpiTS + (threadIdx.x & 31));
        sd = shared;
    }
    __device__ __forceinline__ double rate(double, double hca, double hcb) const { return __dadd_rn(hca, hcb); }
    __device__ __forceinline__ double difference(int i, double d) const {
        const double dy = __dsub_rn(sd[kEpiTS + (threadIdx.x & 31)], sd[(threadIdx.x >> 5) + i * (ET / 32)]);
        if constexpr (ONE) return __fma_rn(from_digit(h[i], t), dy, d);
        else return __fma_rn(h[i], dy, d);
    }
};

template <int STAGE, bool ONE>
__global__ void __launch_bounds__(ET) digits_epi_kernel(DevOps ops, Work w, DigitWork d) {
    extern __shared__ __align__(16) double sm[];
    __shared__ double red[ET / 32], sg[kEpiTS], s_diag[2 * kEpiTS];
    __shared__ int s_done;
    const int I = w.pairs[blockIdx.x].x, J = w.pairs[blockIdx.x].y;
    const bool diag = I == J;
    const int np = ops.np, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t plane = (size_t)np * np;
    double *sX1 = sm, *sX2 = sm + kEpiTS * LDX;
    EpiIn<STAGE, ET> in;
    in.load(ops, w, I, J, d.hc);
    DiagonalTerm<ONE> dg;
    dg.load(ops, d, I, J, s_diag);
    tma::grid_dependency_wait();
    tma::launch_dependents();
    if (threadIdx.x == 0) s_done = *(volatile int *)&w.ctl->done;
#pragma unroll
    for (int a = warp; a < kEpiTS; a += ET / 32) {
        const double *s1 = d.x + (size_t)(I * kEpiTS + a) * np + J * kEpiTS + lane;
        sX1[a * LDX + lane] = __ldcg(s1);
        sX1[a * LDX + kEpiTS + lane] = __ldcg(s1 + plane);
        if (!diag) {
            const double *s2 = d.x + (size_t)(J * kEpiTS + a) * np + I * kEpiTS + lane;
            sX2[a * LDX + lane] = __ldcg(s2);
            sX2[a * LDX + kEpiTS + lane] = __ldcg(s2 + plane);
        }
    }
    if (diag && threadIdx.x < kEpiTS) sg[threadIdx.x] = __ldcg(w.g + I * kEpiTS + threadIdx.x);
    __syncthreads();
    if (s_done) return;
    stage_epilogue<STAGE, ET>(ops, w, I, J, diag, in, sX1, sX2, LDX, sg, red, blockIdx.x, blockIdx.x == 0, dg);
}

template <typename K, typename... A>
void launch_dep(K kernel, int grid, int block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

int gemm_smem(const DigitWork &d) {
    const int ring = d.ring_a * A_BYTES + d.ring_b * d.s * B_ROW;
    return std::max(ring, TM * LDT * (int)sizeof(double)) + 1024;
}

template <int STAGE, int S, int B>
void launch_sb(const DevOps &ops, const Work &w, const DigitWork &d, const DigitMaps &m, cudaStream_t s) {
    const double *yin = (STAGE <= 1) ? w.y : (STAGE == 3 ? w.yb : w.ya);
    launch_dep(split_kernel<S, B>, ops.np, 128, 0, s, ops, w.ctl, yin, d);
    const int tiles = ((ops.np + TM - 1) / TM) * (2 * ops.np / TN);
    launch_dep(digits_gemm_kernel<S, B>, std::max(tiles, d.gain_ctas), GT, (size_t)gemm_smem(d), s, m.h, m.y, ops, w, d, STAGE);
}

template <int STAGE>
void launch_t(const DevOps &ops, const Work &w, const DigitWork &d, const DigitMaps &m, cudaStream_t s) {
    switch (d.b) {
        case 12: launch_sb<STAGE, 6, 12>(ops, w, d, m, s); break;
        case 11: launch_sb<STAGE, 6, 11>(ops, w, d, m, s); break;
        case 10: launch_sb<STAGE, 7, 10>(ops, w, d, m, s); break;
        case 8: launch_sb<STAGE, 8, 8>(ops, w, d, m, s); break;
        case 7: launch_sb<STAGE, 10, 7>(ops, w, d, m, s); break;
        case 6: launch_sb<STAGE, 11, 6>(ops, w, d, m, s); break;
        default: launch_sb<STAGE, 13, 5>(ops, w, d, m, s); break;
    }
    if (d.sh == 1) launch_dep(digits_epi_kernel<STAGE, true>, w.npairs, ET, (size_t)d.epi_smem, s, ops, w, d);
    else launch_dep(digits_epi_kernel<STAGE, false>, w.npairs, ET, (size_t)d.epi_smem, s, ops, w, d);
}

template <bool ONE>
cudaError_t init_epi(int smem) {
    cudaError_t e = raise_smem_limit_t(digits_epi_kernel<0, ONE>, smem);
    if (e == cudaSuccess) e = raise_smem_limit_t(digits_epi_kernel<1, ONE>, smem);
    if (e == cudaSuccess) e = raise_smem_limit_t(digits_epi_kernel<2, ONE>, smem);
    if (e == cudaSuccess) e = raise_smem_limit_t(digits_epi_kernel<3, ONE>, smem);
    if (e == cudaSuccess) e = raise_smem_limit_t(digits_epi_kernel<4, ONE>, smem);
    return e;
}

// The candidates: bits per digit and digits (S b >= 64).
struct Cand {
    int b, s;
};
constexpr Cand kCands[] = {{12, 6}, {11, 6}, {10, 7}, {8, 8}, {7, 10}, {6, 11}, {5, 13}};

}  // namespace

// Digits of H. One digit when every entry is k 2^t with |k| < 2048 (exact in
// FP16); else as many as of Y, of each row by its largest entry. The bits per
// digit are the most for which no sum of a weight's products can leave the
// integers an FP32 accumulator holds exactly: 2^(b-1) times the largest row
// sum of |digits of H| at most 2^24. With unit weights b = 12 up to row sums
// of 8192; with general weights, whose digits are half their largest on
// average, b = 8 for rows of up to about 250 nonzeros, 7 up to 800, 6 up to
// 2900 and 5 up to 10000. Beyond that the FP64 tensor kernel stays in use.
bool plan_digits(const HostOps &h, DigitPlan &p) {
    const int n = (int)h.n;
    if (h.hval.empty()) return false;
    int tmin = 1 << 20, emax = -(1 << 20);
    std::vector<int> etop(n, 0);
    for (int i = 0; i < n; ++i) {
        int et = -(1 << 20);
        for (int64_t q = h.hptr[i]; q < h.hptr[i + 1]; ++q) {
            int e;
            const double f = std::frexp(std::fabs(h.hval[q]), &e);  // f in [1/2, 1)
            const long long m = (long long)std::ldexp(f, 53);
            tmin = std::min(tmin, e - 53 + __builtin_ctzll((unsigned long long)m));
            et = std::max(et, e);
        }
        if (et == -(1 << 20)) et = 0;
        etop[i] = et;
        emax = std::max(emax, et);
    }
    // a tiny or huge scale would leave the exponent range of the products
    if (emax > 400 || tmin < -700) return false;
    const bool one = emax - tmin <= 11;  // |k| < 2^11
    for (const Cand &c : kCands) {
        if (!one && c.b > 8) continue;
        const int sh = one ? 1 : c.s;
        double worst = 0.0;
        p.erow.assign(n, 0);
        for (int i = 0; i < n; ++i) {
            p.erow[i] = one ? tmin : etop[i] - (c.b - 1);
            double l1 = 0.0;
            for (int64_t q = h.hptr[i]; q < h.hptr[i + 1]; ++q) {
                int16_t d[kMaxDigits];
                digits_of(h.hval[q], p.erow[i] - c.b * (sh - 1), sh, c.b, d);
                for (int s = 0; s < sh; ++s) l1 += std::fabs((double)d[s]);
            }
            worst = std::max(worst, l1);
        }
        if (worst * (double)(1 << (c.b - 1)) > 16777216.0) continue;
        p.b = c.b;
        p.s = c.s;
        p.sh = sh;
        return true;
    }
    return false;
}

size_t digits_half_count(const DigitPlan &p, int np) { return (size_t)(p.sh + 2 * p.s) * np * np; }
size_t digits_double_count(const DigitPlan &p, int np) { return (size_t)(p.sh > 1 ? 3 : 2) * np * np + 2 * (size_t)np; }

cudaError_t init_digits(const DevOps &ops, const DigitPlan &p, int sms, void *halves, int *ints, double *x, DigitWork *dw,
                        DigitMaps *maps) {
    const int np = ops.np;
    const size_t plane = (size_t)np * np;
    __half *hd = reinterpret_cast<__half *>(halves);
    dw->yd = hd + p.sh * plane;
    dw->ecol = ints;
    dw->erow = ints + 2 * np;
    dw->x = x;
    dw->diag = x + 2 * plane;
    dw->hd = hd;
    double *hc = x + 2 * plane + np, *hf = hc + np;
    dw->hc = hc;
    dw->h = hf;
    dw->unit = p.erow[0];
    dw->b = p.b;
    dw->s = p.s;
    dw->sh = p.sh;
    dw->tmem_cols = p.s * TN <= 256 ? 256 : 512;
    const int tiles = ((np + TM - 1) / TM) * (2 * np / TN);
    dw->gain_ctas = std::max(std::min(sms, tiles), std::min(sms, (np + GT / 32 - 3) / (GT / 32 - 2)));  // a row per warp
    // The epilogue's CTAs become resident while the product still runs, on
    // whatever SMs have room: 136 of them piled up on the 24 SMs without a
    // product CTA at N = 500 (12.6 us against 4.5 for three). Where a CTA per
    // SM will do, each asks for more than half of an SM's shared memory.
    dw->epi_smem = ops.np / kEpiTS * (ops.np / kEpiTS + 1) / 2 <= sms ? 116 * 1024 : EPI_BYTES;
    // rings: all of an SM when there is a tile per SM at most, else half of it,
    // for two CTAs; with S >= 10 a CTA holds all of TMEM, so only one of them
    // works, and at S = 11 and 13 the smallest rings are above the half (121
    // and 137 KB)
    const int room = (tiles <= sms ? 200 : 96) * 1024;
    dw->ring_b = std::max(2, std::min(kMaxRing, room / (A_BYTES + p.s * B_ROW)));
    if (p.sh > 1) dw->ring_b = 2;
    dw->ring_a = std::max(2, std::min(kMaxRing, (room - dw->ring_b * p.s * B_ROW) / A_BYTES));
    cudaError_t e = cudaMemset(halves, 0, digits_half_count(p, np) * sizeof(__half));
    if (e != cudaSuccess) return e;
    e = cudaMemcpy(dw->erow, p.erow.data(), p.erow.size() * sizeof(int), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return e;
    if (p.sh > 1) e = cudaMemset(hf, 0, plane * sizeof(double));
    if (e != cudaSuccess) return e;
    split_h_kernel<<<std::min(ops.n, 4096), 128>>>(ops, p.b, p.sh, dw->erow, hd, hf, hc);
    e = cudaStreamSynchronize(nullptr);
    if (e != cudaSuccess) return e;
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;
    const cuuint64_t n64 = (cuuint64_t)np;
    cuuint32_t es[4] = {1, 1, 1, 1};
    {
        cuuint64_t dims[3] = {n64, n64, (cuuint64_t)p.sh}, strides[2] = {n64 * 2, n64 * n64 * 2};
        cuuint32_t box[3] = {BK, TM, 1};
        if (enc(&maps->h, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, hd, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    {
        cuuint64_t dims[4] = {n64, n64, 2, (cuuint64_t)p.s}, strides[3] = {n64 * 2, n64 * n64 * 2, 2 * n64 * n64 * 2};
        cuuint32_t box[4] = {BK, TN, 1, (cuuint32_t)p.s};
        if (enc(&maps->y, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, dw->yd, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    const int sm = gemm_smem(*dw);
    switch (p.b) {
        case 12: e = raise_smem_limit_t(digits_gemm_kernel<6, 12>, sm); break;
        case 11: e = raise_smem_limit_t(digits_gemm_kernel<6, 11>, sm); break;
        case 10: e = raise_smem_limit_t(digits_gemm_kernel<7, 10>, sm); break;
        case 8: e = raise_smem_limit_t(digits_gemm_kernel<8, 8>, sm); break;
        case 7: e = raise_smem_limit_t(digits_gemm_kernel<10, 7>, sm); break;
        case 6: e = raise_smem_limit_t(digits_gemm_kernel<11, 6>, sm); break;
        default: e = raise_smem_limit_t(digits_gemm_kernel<13, 5>, sm); break;
    }
    if (e == cudaSuccess) e = p.sh == 1 ? init_epi<true>(dw->epi_smem) : init_epi<false>(dw->epi_smem);
    return e;
}

void launch_stage_digits(int stage, const DevOps &ops, const Work &w, const DigitWork &d, const DigitMaps &m, cudaStream_t s) {
    switch (stage) {
        case 0: launch_t<0>(ops, w, d, m, s); break;
        case 1: launch_t<1>(ops, w, d, m, s); break;
        case 2: launch_t<2>(ops, w, d, m, s); break;
        case 3: launch_t<3>(ops, w, d, m, s); break;
        default: launch_t<4>(ops, w, d, m, s); break;
    }
}

}  // namespace qpr
