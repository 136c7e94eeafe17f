// Classical PageRank and hub classes (main text, the airline ranking: the
// quantum PageRank populations compared with the classical PageRank vector,
// nodes sorted into main and secondary hubs).
//
// The classical PageRank is the stationary vector pi of the Google matrix
// G = alpha S + (1 - alpha) F (Eq. S4 with the column-normalised adjacency,
// F of Eq. S2): G pi = pi, sum pi = 1. It is also the populations of the
// omega = 1 steady state of the Lindblad equation (Eq. 1 with only the
// dissipator, whose populations follow dp/dt = G p - c o p with c = 1).
// Power iteration pi <- G pi from the uniform vector, in FP64: each
// iteration is one kernel whose CTAs form G pi for their rows (CSR of S,
// the dangling columns, the teleport part) and per-CTA partials of the L1
// change, which the host sums in index order every few iterations.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

#include "gain_body.cuh"
#include "qpr_internal.cuh"

namespace qpr {
namespace {

constexpr int kPrThreads = 256;

using gain64::block_sum;

// One power-iteration step: out = G pi / sum(pi) for rows of this CTA
// (rows blk, blk + grid, ... in warps), and this CTA's partial of
// sum |out_i - pi_i| / sum(pi) (delta[blk]). Every CTA sums pi and its
// dangling part itself, in the same order, so the iteration is
// deterministic.
__global__ void __launch_bounds__(kPrThreads) pagerank_step_kernel(DevOps ops, const double *__restrict__ pi,
                                                                  double *__restrict__ out,
                                                                  double *__restrict__ delta) {
    __shared__ double red[32];
    const int n = ops.n;
    double P = 0.0, Dd = 0.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const double pj = pi[j];
        P += pj;
        if (ops.dang[j]) Dd += pj;
    }
    P = block_sum(P, red);
    Dd = block_sum(Dd, red);
    const double inv = 1.0 / P;
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    double dl = 0.0;
    for (int i = blockIdx.x * warps + (threadIdx.x >> 5); i < n; i += gridDim.x * warps) {
        double s = 0.0;
        for (int q = ops.s_ptr[i] + lane; q < ops.s_ptr[i + 1]; q += 32) s += ops.s_val[q] * pi[ops.s_col[q]];
        s = gain64::warp_sum(s);
        if (lane == 0) {
            const double pii = pi[i];
            const double dterm = (ops.dangling == QPR_DANGLING_F) ? (Dd - (ops.dang[i] ? pii : 0.0)) / (n - 1)
                                                                  : Dd / n;
            const double g = (ops.alpha * (s + dterm) + (1.0 - ops.alpha) * (P - pii) / (n - 1)) * inv;
            out[i] = g;
            dl += fabs(g - pii * inv);
        }
    }
    dl = block_sum(dl, red);
    if (threadIdx.x == 0) delta[blockIdx.x] = dl;
}

// Power iteration by one cluster of 8 CTAs, the iterate in every CTA's shared
// memory (two buffers), thousands of iterations per launch. A launch per
// iteration took 8 us at N = 922, most of it latency, with a wait for the
// host every eighth one. What bounds an iteration here is its chain of FP64
// instructions (40 ns each on a scheduler) and one cluster barrier, 3 us, so
// it has as few as can be: the columns of G sum to one, so sum(pi) stays 1
// and the teleport part (1 - alpha) (1 - pi_i) / (N - 1) needs no sum and no
// division (rounding in the sum decays by alpha per iteration; the result is
// normalised once). Four lanes sum a row of S (a warp one of more than kPrLong
// entries), four warps the dangling nodes if there are any, then a thread per
// row writes the new entry into all 8 copies through distributed shared
// memory.
constexpr int kPrCtas = 8;
constexpr int kPrT = 512;
constexpr int kPrLong = 48;

__device__ __forceinline__ uint32_t pr_remote(const void *p, int cta) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n"
                 : "=r"(r)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(cta));
    return r;
}
__device__ __forceinline__ void pr_store(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;\n" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void pr_barrier() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
size_t pr_smem(int n) { return (size_t)(2 * n + (n + kPrCtas - 1) / kPrCtas) * sizeof(double) + n; }

// jobs[blockIdx.y]. state (null: none): {iterations done, last L1 change, 1 if
// stopped}; with it the iterate is kept in `pi` between launches (start: the
// uniform vector when no iteration is done), and the L1 change is formed at
// every eighth iteration and at max_iter, where the run stops (below tol, not
// finite, or max_iter).
__global__ void __cluster_dims__(kPrCtas, 1, 1) __launch_bounds__(kPrT, 1)
pagerank_cluster_kernel(const PrJob *__restrict__ jobs, PrJob one, int iters, double tol, long long max_iter,
                        double *state) {
    extern __shared__ __align__(16) double sm[];
    // the CTAs' parts of the L1 change, one copy for every other iteration: a
    // limit of 8 m + 1 makes two checks follow each other with one barrier
    // between, and a CTA may still read the first while a peer stores the second
    __shared__ double s_part[4], s_dang, s_delta[2][kPrCtas], red[32];
    const PrJob g = jobs ? jobs[blockIdx.y] : one;
    const int n = g.n, cta = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (n + kPrCtas - 1) / kPrCtas, r0 = min(n, cta * per), rows = min(n, r0 + per) - r0;
    double *rowsum = sm + 2 * n;
    unsigned char *dang = reinterpret_cast<unsigned char *>(rowsum + per);
    const bool resume = state && state[0] > 0.0;
    int any = 0;
    for (int i = tid; i < n; i += kPrT) {
        sm[i] = resume ? g.pi[i] : 1.0 / n;
        dang[i] = g.dang[i];
        any = any || dang[i];
    }
    any = __syncthreads_or(any);
    if (tid == 0) s_dang = 0.0;
    long long it = state ? (long long)state[0] : 0;
    const double inv_nm1 = 1.0 / (double)(n - 1), inv_n = 1.0 / (double)n;
    const double tele = (1.0 - g.alpha) * inv_nm1;
    __syncthreads();
    pr_barrier();  // the cluster's CTAs run, and have read the state
    int cur = 0;
    bool stopped = false;
    double delta = 0.0;
    for (int k = 0; k < iters && !stopped; ++k) {
        const double *pi = sm + (size_t)cur * n;
        double *nx = sm + (size_t)(1 - cur) * n;
        if (any && warp < 4) {
            double D = 0.0;
            for (int j = tid; j < n; j += 128)
                if (dang[j]) D += pi[j];
            D = gain64::warp_sum(D);
            if (lane == 0) s_part[warp] = D;
            asm volatile("bar.sync 1, 128;\n" ::: "memory");
            if (tid == 0) s_dang = (s_part[0] + s_part[1]) + (s_part[2] + s_part[3]);
        }
        // quads: 8 rows of this CTA per warp and pass
        for (int b = warp * 8; b < rows; b += (kPrT / 32) * 8) {
            const int i = b + (lane >> 2);
            int q0 = 0, q1 = 0;
            if (i < rows) {
                q0 = g.s_ptr[r0 + i];
                q1 = g.s_ptr[r0 + i + 1];
            }
            const bool lng = q1 - q0 > kPrLong;
            double s = 0.0;
            if (!lng)
                for (int q = q0 + (lane & 3); q < q1; q += 4) s += g.s_val[q] * pi[g.s_col[q]];
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (!lng && (lane & 3) == 0 && i < rows) rowsum[i] = s;
            for (unsigned m = __ballot_sync(0xffffffffu, lng && (lane & 3) == 0); m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                const int a0 = __shfl_sync(0xffffffffu, q0, src), a1 = __shfl_sync(0xffffffffu, q1, src);
                double t = 0.0;
                for (int q = a0 + lane; q < a1; q += 32) t += g.s_val[q] * pi[g.s_col[q]];
                t = gain64::warp_sum(t);
                if (lane == 0) rowsum[b + (src >> 2)] = t;
            }
        }
        __syncthreads();
        ++it;
        const bool check = state && (it % 8 == 0 || it >= max_iter);
        const double D = s_dang;
        double dl = 0.0;
        for (int i = tid; i < rows; i += kPrT) {
            const int gi = r0 + i;
            const double p = pi[gi];
            double s = rowsum[i];
            if (any) s += (g.dangling == QPR_DANGLING_F) ? (D - (dang[gi] ? p : 0.0)) * inv_nm1 : D * inv_n;
            const double v = g.alpha * s + tele * (1.0 - p);
            for (int c = 0; c < kPrCtas; ++c) pr_store(pr_remote(nx + gi, c), v);
            if (check) dl += fabs(v - p);
        }
        if (check) {
            dl = block_sum(dl, red);
            if (tid < kPrCtas) pr_store(pr_remote(&s_delta[cur][cta], tid), dl);
        }
        pr_barrier();
        cur = 1 - cur;
        if (check) {
            delta = 0.0;
            for (int c = 0; c < kPrCtas; ++c) delta += s_delta[1 - cur][c];
            stopped = !(delta >= tol) || it >= max_iter;  // the same in every CTA
        }
    }
    const double *pi = sm + (size_t)cur * n;
    double P = 0.0;
    if (!state || stopped) {  // normalised result
        for (int j = tid; j < n; j += kPrT) P += pi[j];
        P = block_sum(P, red);
    } else {
        P = 1.0;
    }
    for (int i = tid; i < rows; i += kPrT) {
        const double v = pi[r0 + i] / P;
        if (g.pi) g.pi[r0 + i] = v;
        if (g.feature) g.feature[(size_t)(r0 + i) * g.stride] = (float)log((double)n * v);
    }
    if (state && cta == 0 && tid == 0) {
        state[0] = (double)it;
        state[1] = delta;
        state[2] = stopped ? 1.0 : 0.0;
    }
}

__global__ void uniform_kernel(double *pi, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) pi[i] = 1.0 / n;
}

// pi / sum(pi) into out (one CTA; fixed-order sum).
__global__ void __launch_bounds__(1024) normalize_kernel(const double *__restrict__ pi, int n,
                                                         double *__restrict__ out) {
    __shared__ double red[32];
    double P = 0.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) P += pi[j];
    P = block_sum(P, red);
    for (int j = threadIdx.x; j < n; j += blockDim.x) out[j] = pi[j] / P;
}

// classes[i] = 2 (main hub, p_i > c / N), 1 (secondary, 1/N < p_i <= c/N),
// 0 otherwise; counts[k] += the nodes of class k.
__global__ void hub_kernel(const double *__restrict__ p, int n, double c, int *__restrict__ classes,
                           unsigned long long *__restrict__ counts) {
    __shared__ unsigned int cnt[3];
    if (threadIdx.x < 3) cnt[threadIdx.x] = 0;
    __syncthreads();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double v = p[i];
        const int k = (v > c / (double)n) ? 2 : (v > 1.0 / (double)n ? 1 : 0);
        classes[i] = k;
        atomicAdd(&cnt[k], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 3) atomicAdd(&counts[threadIdx.x], (unsigned long long)cnt[threadIdx.x]);
}

}  // namespace

int pagerank_grid(int n) {
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
        cudaGetLastError();
        sms = 1;
    }
    const int rows_per_cta = kPrThreads / 32;
    int grid = (n + rows_per_cta - 1) / rows_per_cta;
    if (grid > 2 * sms) grid = 2 * sms;
    return grid < 1 ? 1 : grid;
}

cudaError_t pagerank(const DevOps &ops, double tol, int64_t max_iter, double *scratch, double *pi_out_dev,
                     int64_t *iters, double *delta_out, cudaStream_t s) {
    const int n = ops.n;
    const int grid = pagerank_grid(n);
    cudaError_t e = cudaSuccess;
    double *a = scratch, *b = scratch + n, *delta = scratch + 2 * (size_t)n;
    uniform_kernel<<<(n + 255) / 256, 256, 0, s>>>(a, n);
    std::vector<double> part(grid);
    // check convergence every `chunk` iterations (the host reads the last
    // iteration's partials)
    const int chunk = 8;
    int64_t it = 0;
    double d = INFINITY;
    while (it < max_iter) {
        const int64_t k1 = std::min<int64_t>(max_iter, it + chunk);
        for (; it < k1; ++it) {
            pagerank_step_kernel<<<grid, kPrThreads, 0, s>>>(ops, a, b, delta);
            std::swap(a, b);
        }
        e = cudaMemcpyAsync(part.data(), delta, grid * sizeof(double), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) break;
        d = 0.0;
        for (double v : part) d += v;
        if (!(d >= tol)) break;  // converged (or not finite)
    }
    if (e == cudaSuccess) {
        normalize_kernel<<<1, 1024, 0, s>>>(a, n, pi_out_dev);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (iters) *iters = it;
    if (delta_out) *delta_out = d;
    return e;
}

// Which form: the cluster has 32 schedulers, the grid up to 1216 but a launch
// per iteration and the sums over all nodes in every CTA. Per iteration the
// cluster takes about 3 us and 10.5 ns for each FP64 warp instruction of its
// busiest CTA (counted below from the rows' lengths), the grid 13 us and 4.5 ns
// per node. Measured, cluster against grid, us per iteration: sparse
// (heavy-tailed, 8 links a node) N = 922 3.2 and 14.6, N = 8192 15.6 and 48;
// links with p = 0.25 N = 700 12.1 and 15.6, N = 900 18.5 and 16.0, N = 2000 68
// and 27, N = 4000 181 and 43; p = 0.005 N = 8192 35 and 49; 60 rows of all
// nodes N = 2000 39 and 28. The cluster form also takes the columns of S to
// sum to one, which they do unless an out-degree overflows.
bool pagerank_in_cluster(const HostOps &h) {
    const int n = (int)h.n;
    if (n > kPrClusterMaxN) return false;
    for (double d : h.outdeg)
        if (!std::isfinite(d)) return false;
    const int per = (n + kPrCtas - 1) / kPrCtas;
    int64_t most = 0;
    for (int r0 = 0; r0 < n; r0 += per) {
        const int r1 = std::min(n, r0 + per);
        int64_t work = 6 * ((r1 - r0 + 31) / 32);
        for (int b = r0; b < r1; b += 8) {
            int quad = 0;  // rounds of the longest short row of a warp's eight
            for (int i = b; i < std::min(r1, b + 8); ++i) {
                const int len = h.sptr[i + 1] - h.sptr[i];
                if (len > kPrLong) work += (len + 31) / 32 + 5;
                else quad = std::max(quad, (len + 3) / 4);
            }
            work += quad + 2;
        }
        most = std::max(most, work);
    }
    return (double)most <= 950.0 + 0.43 * n;
}

cudaError_t pagerank_cluster(const DevOps &ops, double tol, int64_t max_iter, double *scratch, double *pi_out_dev,
                             int64_t *iters, double *delta_out, int64_t *launches, cudaStream_t s) {
    const int n = ops.n;
    PrJob job{};
    job.n = n;
    job.dangling = ops.dangling;
    job.alpha = ops.alpha;
    job.s_ptr = ops.s_ptr;
    job.s_col = ops.s_col;
    job.s_val = ops.s_val;
    job.dang = ops.dang;
    job.pi = scratch;
    double *state = scratch + n;
    cudaError_t e = raise_smem_limit_t(pagerank_cluster_kernel, (int)pr_smem(n));
    if (e == cudaSuccess) e = cudaMemsetAsync(state, 0, kPrState * sizeof(double), s);
    double h[kPrState] = {0.0, INFINITY, 0.0, 0.0};
    *launches = 0;
    while (e == cudaSuccess && h[2] == 0.0) {
        pagerank_cluster_kernel<<<kPrCtas, kPrT, pr_smem(n), s>>>(nullptr, job, 4096, tol, (long long)max_iter, state);
        ++*launches;
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(h, state, sizeof(h), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(pi_out_dev, scratch, n * sizeof(double), cudaMemcpyDeviceToDevice, s);
    if (iters) *iters = (int64_t)h[0];
    if (delta_out) *delta_out = h[1];
    return e;
}

cudaError_t pagerank_jobs(const PrJob *jobs, int count, int max_n, int iters, cudaStream_t s) {
    cudaError_t e = raise_smem_limit_t(pagerank_cluster_kernel, (int)pr_smem(max_n));
    if (e != cudaSuccess) return e;
    for (int at = 0; at < count; at += 32768)
        pagerank_cluster_kernel<<<dim3(kPrCtas, std::min(count - at, 32768)), kPrT, pr_smem(max_n), s>>>(
            jobs + at, PrJob{}, iters, 0.0, 0, nullptr);
    return cudaGetLastError();
}

cudaError_t hub_classes(const double *p, int n, double c, int *classes_dev, unsigned long long *counts_dev,
                        cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(counts_dev, 0, 3 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    int grid = (n + 255) / 256;
    if (grid > 1024) grid = 1024;
    hub_kernel<<<grid, 256, 0, s>>>(p, n, c, classes_dev, counts_dev);
    return cudaGetLastError();
}

}  // namespace qpr
