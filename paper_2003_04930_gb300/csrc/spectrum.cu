// Spectral spread of H: power iteration for its eigenvalue of largest modulus
// l1, then for that of H - l1 I (the far end of the spectrum), 400 products
// each, one cluster of 8 CTAs per matrix.
//
// On the host this was most of a context's set-up (800 sweeps over the
// nonzeros: qpr_create 10.3 ms at N = 922, 196 ms at N = 900 with 394 nonzeros
// a row; 6.4 and 34 with this). What bounds it here is the chain of a product:
// a row's FP64 sum and one cluster barrier, 3.7 us at N = 300 and 4.2 at 922.
// So the vector stays in every CTA's shared memory (two buffers, entries
// written through distributed shared memory), four lanes sum a row (a warp one
// of more than kLong entries), the vector is rescaled by its norm only at every
// eighth product, and the Rayleigh quotient is formed at the last one.
#include <math.h>

#include <algorithm>

#include "gain_body.cuh"
#include "qpr_internal.cuh"

namespace qpr {
namespace {

constexpr int kCtas = 8;
constexpr int kT = 512;
constexpr int kLong = 48;
constexpr int kProducts = 400;

__device__ __forceinline__ void put(const double *p, int cta, double v) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(cta));
    asm volatile("st.shared::cluster.f64 [%0], %1;\n" ::"r"(r), "d"(v) : "memory");
}
__device__ __forceinline__ void barrier() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

size_t spectrum_smem(int n) { return (size_t)2 * n * sizeof(double); }

__global__ void __cluster_dims__(kCtas, 1, 1) __launch_bounds__(kT, 1)
spectrum_kernel(const SpectrumJob *__restrict__ jobs, SpectrumJob one) {
    extern __shared__ __align__(16) double sm[];
    __shared__ double s_dot[kCtas][2], red[32];
    const SpectrumJob g = jobs ? jobs[blockIdx.y] : one;
    const int n = g.n, cta = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (n + kCtas - 1) / kCtas, r0 = min(n, cta * per), rows = min(n, r0 + per) - r0;
    barrier();  // the cluster's CTAs run
    double shift = 0.0, lam = 0.0;
    for (int pass = 0; pass < 2; ++pass) {
        for (int i = tid; i < n; i += kT) sm[i] = 1.0 + 0.37 * sin(0.7 * (double)i + 0.1);
        __syncthreads();
        double scale = 1.0;  // of the stored vector at its next use
        lam = 0.0;
        for (int it = 0; it < kProducts; ++it) {
            const double *x = sm + (size_t)(it & 1) * n;
            const double *y = sm + (size_t)(1 - (it & 1)) * n;
            const bool norm = (it & 7) == 7 || it == kProducts - 1;
            double xx = 0.0, xz = 0.0;
            auto row_done = [&](int i, double s) {  // one lane
                const double xi = x[r0 + i] * scale;
                const double z = __fma_rn(-shift, xi, s * scale);
                if (norm) {
                    xx = __fma_rn(xi, xi, xx);
                    xz = __fma_rn(xi, z, xz);
                }
                for (int c = 0; c < kCtas; ++c) put(y + r0 + i, c, z);
            };
            for (int b = warp * 8; b < rows; b += (kT / 32) * 8) {
                const int i = b + (lane >> 2);
                int q0 = 0, q1 = 0;
                if (i < rows) {
                    q0 = g.h_ptr[r0 + i];
                    q1 = g.h_ptr[r0 + i + 1];
                }
                const bool lng = q1 - q0 > kLong;
                double s = 0.0;
                if (!lng)
                    for (int q = q0 + (lane & 3); q < q1; q += 4) s = __fma_rn(g.h_val[q], x[g.h_col[q]], s);
                s += __shfl_xor_sync(0xffffffffu, s, 1);
                s += __shfl_xor_sync(0xffffffffu, s, 2);
                if (!lng && (lane & 3) == 0 && i < rows) row_done(i, s);
                for (unsigned m = __ballot_sync(0xffffffffu, lng && (lane & 3) == 0); m; m &= m - 1) {
                    const int src = __ffs(m) - 1;
                    const int a0 = __shfl_sync(0xffffffffu, q0, src), a1 = __shfl_sync(0xffffffffu, q1, src);
                    double t = 0.0;
                    for (int q = a0 + lane; q < a1; q += 32) t = __fma_rn(g.h_val[q], x[g.h_col[q]], t);
                    t = gain64::warp_sum(t);
                    if (lane == 0) row_done(b + (src >> 2), t);
                }
            }
            if (norm) {
                xx = gain64::block_sum(xx, red);
                xz = gain64::block_sum(xz, red);
                if (tid < kCtas) {
                    put(&s_dot[cta][0], tid, xx);
                    put(&s_dot[cta][1], tid, xz);
                }
            }
            barrier();
            scale = 1.0;
            if (norm) {
                double a = 0.0, b = 0.0;
                for (int c = 0; c < kCtas; ++c) {
                    a += s_dot[c][0];
                    b += s_dot[c][1];
                }
                if (a == 0.0) {  // H = 0
                    lam = 0.0;
                    break;
                }
                lam = b / a;
                scale = 1.0 / sqrt(a);
                __syncthreads();  // s_dot is written again at the earliest after the next barrier
            }
        }
        shift = lam;
        __syncthreads();
        barrier();  // the buffers are filled anew
    }
    if (cta == 0 && tid == 0) *g.out = fabs(lam) * 1.02 + 1e-12;
}

}  // namespace

cudaError_t spectral_spread(const SpectrumJob *jobs, int count, int max_n, const SpectrumJob &one, cudaStream_t s) {
    cudaError_t e = raise_smem_limit_t(spectrum_kernel, (int)spectrum_smem(max_n));
    if (e != cudaSuccess) return e;
    if (!jobs) {
        spectrum_kernel<<<kCtas, kT, spectrum_smem(max_n), s>>>(nullptr, one);
        return cudaGetLastError();
    }
    for (int at = 0; at < count; at += 32768)
        spectrum_kernel<<<dim3(kCtas, std::min(count - at, 32768)), kT, spectrum_smem(max_n), s>>>(jobs + at, one);
    return cudaGetLastError();
}

}  // namespace qpr
