// FP64 RK4 of a small problem (N <= kSmallMaxN) as one persistent launch of
// one cluster of 8 CTAs: a whole block of steps, no kernel boundary in it.
//
// What bounds it: a step of a small problem is a chain of four dependent
// stages of a few thousand FP64 operations; as eight launches a step (gain
// and stage kernel per stage) it cost 139 us at N = 16 and 366 us at N = 44,
// all of it launch latency and one CTA's serial chain through a 32 x 32
// tile; now 7.5 us at N = 16, 23 at N = 32 and 39 at N = 44 (Erdos-Renyi, p = 0.25). Here the state stays on chip. FP64 runs at two operations a clock
// and SM, so one warp instruction holds its scheduler for about 64 clocks:
// what counts is the number of FP64 instructions in sequence on a scheduler,
// not the threads in flight. So a lane octet owns one element (a, b), a <= b, of
// the Hermitian state for the whole launch (its y and RK4 sum in registers):
// the octet's lanes share the two sparse rows of
//     k_ab = (1 - omega) [ (B_ab + B_ba) - i (A_ab - A_ba) ] + ...,
//     A = H Re Y, B = H Im Y,
// the first reduction step leaves the real part in the even lanes and the
// imaginary part in the odd ones, and both run the rest in the same
// instructions. Elements go round the 8 SMs warp by warp. Every CTA keeps the
// whole stage input (two buffers) in its shared memory; an element's lanes
// write the next input and its mirror image into all 8 copies through
// distributed shared memory, and one cluster barrier ends the stage.
//
// Off the elements' chain, one more warp per CTA sums the trace of y during
// stage 1 (the step is linear, so 1 / tr(y) is applied once, at stage 4)
// and, during stage 3, the residual partials of stage 1, in index order, so
// that all CTAs take the same stop decision with no message. y changes only
// at stage 4, so a run that stops at step n still holds y_n.
#include <math.h>

#include "qpr_internal.cuh"

namespace qpr {
namespace {

constexpr int kCtas = 8;       // one cluster
constexpr int kOctets = 4;     // elements per warp

__device__ __forceinline__ uint32_t remote_addr(const void *p, int cta) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(a), "r"(cta));
    return r;
}
__device__ __forceinline__ void remote_store(uint32_t addr, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;\n" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ double xor_add(double v, int o) { return v + __shfl_xor_sync(0xffffffffu, v, o); }

__host__ __device__ constexpr int small_ld(int n) { return n | 1; }

// Runs up to `limit` steps from the state in w.y (or until the stop rule
// sets ctl->done) and writes the state back. `warps`: element warps per CTA;
// the block has one more.
__global__ void __launch_bounds__(1024, 1) small_rk4_kernel(DevOps ops, Work w, int warps, int nnz, int limit) {
    extern __shared__ __align__(16) double smem[];
    __shared__ double s_scale, s_trace;
    __shared__ int s_stop;
    Ctl *ctl = w.ctl;
    const int n = ops.n, np = ops.np, ld = small_ld(n);
    const size_t plane = (size_t)np * np;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cta = blockIdx.x;  // the grid is one cluster
    const int sz = n * ld;
    double *buf = smem;             // [2 buffers][Re, Im][n][ld]
    double *G = buf + 4 * sz;       // the Google matrix
    double *hval = G + sz;
    double *part = hval + nnz;      // residual partials of all element warps
    int *hptr = reinterpret_cast<int *>(part + kCtas * warps);
    int *hcol = hptr + n + 1;
    const int done = *(volatile int *)&ctl->done;
    long long step = *(volatile long long *)&ctl->step;
    const long long max_steps = ctl->max_steps;
    const double tol = ctl->tol, dt = ctl->dt;

    for (int t = tid; t < n * n; t += blockDim.x) {
        const int a = t / n, b = t - a * n;
        buf[a * ld + b] = w.y[(size_t)a * np + b];
        buf[sz + a * ld + b] = w.y[plane + (size_t)a * np + b];
        // G = alpha S + (1 - alpha) F; a dangling column of S is F's column or uniform
        const double f = (a == b) ? 0.0 : 1.0 / (double)(n - 1);
        double s = 0.0;
        if (ops.dang[b]) {
            s = (ops.dangling == QPR_DANGLING_F) ? f : 1.0 / (double)n;
        } else {
            for (int q = ops.s_ptr[a]; q < ops.s_ptr[a + 1]; ++q)
                if (ops.s_col[q] == b) s = ops.s_val[q];
        }
        G[a * ld + b] = ops.alpha * s + (1.0 - ops.alpha) * f;
    }
    for (int t = tid; t < nnz; t += blockDim.x) {
        hval[t] = ops.h_val[t];
        hcol[t] = ops.h_col[t];
    }
    for (int t = tid; t <= n; t += blockDim.x) hptr[t] = ops.h_ptr[t];
    if (tid == 0) s_stop = 0;
    __syncthreads();
    // every CTA of the cluster runs (its shared memory may be written) and has read ctl
    cluster_arrive();
    cluster_wait();
    if (done) return;

    const bool element_warp = warp < warps;
    const int gw = warp * kCtas + cta;  // element warps go round the CTAs
    const int l = lane & 7;
    const bool even = (l & 1) == 0;
    const int total = n * (n + 1) / 2;
    const int e = gw * kOctets + (lane >> 3);
    const bool own = element_warp && e < total;
    int a = 0, b = 0;
    if (own) {
        if (e < n) {
            a = b = e;  // the diagonal first: its warps also form the gain
        } else {
            int r = e - n;
            while (r >= n - 1 - a) {
                r -= n - 1 - a;
                ++a;
            }
            b = a + 1 + r;
        }
    }
    const bool diag = a == b;
    const bool diag_warp = element_warp && gw * kOctets < n;
    const int pa = own ? hptr[a] : 0, na = own ? hptr[a + 1] - pa : 0;
    const int pb = own ? hptr[b] : 0, nb = own ? hptr[b + 1] - pb : 0;
    const double om = ops.omega, cm = 1.0 - om;
    const double csign = even ? cm : -cm;
    const double hc = own ? om * (0.5 * (ops.c[a] + ops.c[b])) : 0.0;
    const double dt2 = 0.5 * dt, dt3 = dt / 3.0, dt6 = dt / 6.0;
    const double weight = (own && l < 2) ? (diag ? 1.0 : 2.0) : 0.0;
    double y = own ? buf[(even ? 0 : sz) + a * ld + b] : 0.0;  // this lane's component of y_ab
    double z = 0.0, cur = y, nrm = 0.0;
    double scale = 1.0, P = 0.0;  // last warp
    // the two copies this lane writes the next input to: its component of (a, b) and of (b, a)
    const uint32_t base0 = remote_addr(buf, l & 6), base1 = remote_addr(buf, (l & 6) + 1);
    const uint32_t oab = (uint32_t)(((even ? 0 : sz) + a * ld + b) * sizeof(double));
    const uint32_t oba = (uint32_t)(((even ? 0 : sz) + b * ld + a) * sizeof(double));
    const uint32_t bufbytes = (uint32_t)(2 * sz * sizeof(double));

    // k of this lane's component for the stage input in buffer `in`
    auto rhs = [&](const double *R, const double *I) {
        double accA = 0.0, accB = 0.0;
        for (int t = l; t < na + nb; t += 8) {
            const bool row_a = t < na;
            const int q = row_a ? pa + t : pb + (t - na);
            const int o = hcol[q] * ld + (row_a ? b : a);
            const double h = hval[q];
            accA = __fma_rn(row_a ? h : -h, R[o], accA);
            accB = __fma_rn(h, I[o], accB);
        }
        // even lanes take B_ab + B_ba, odd lanes A_ab - A_ba
        double x = (even ? accB : accA) + __shfl_xor_sync(0xffffffffu, even ? accA : accB, 1);
        x = xor_add(x, 2);
        x = xor_add(x, 4);
        double k = __fma_rn(-hc, cur, csign * x);
        if (diag_warp) {
            double g = 0.0;
            if (own && diag)
                for (int j = l; j < n; j += 8) g = __fma_rn(G[a * ld + j], R[j * ld + j], g);
            g = xor_add(g, 1);
            g = xor_add(g, 2);
            g = xor_add(g, 4);
            if (diag) k = even ? __fma_rn(om, g, k) : 0.0;
        }
        return k;
    };
    auto publish = [&](int out) {
        if (own) {
            const uint32_t o = out ? bufbytes : 0;
            const double m = even ? cur : -cur;
            remote_store(base0 + o + oab, cur);
            remote_store(base1 + o + oab, cur);
            if (!diag) {
                remote_store(base0 + o + oba, m);
                remote_store(base1 + o + oba, m);
            }
        }
        __syncwarp();
        cluster_arrive();
    };

    int ran = 0;
    bool stopped = false;
    for (;;) {
        // stage 1: buffer 0 -> 1
        if (element_warp) {
            const double k = rhs(buf, buf + sz);
            z = __fma_rn(dt6, k, y);
            cur = __fma_rn(dt2, k, y);
            nrm = weight * k * k;
        } else {
            for (int j = lane; j < n; j += 32) P = (j < 32) ? buf[j * ld + j] : P + buf[j * ld + j];
            if (lane >= n) P = 0.0;
            for (int o = 16; o > 0; o >>= 1) P = xor_add(P, o);
            scale = 1.0 / P;
            if (lane == 0) {
                s_scale = scale;
                s_trace = P;
            }
        }
        publish(1);
        if (element_warp) {
            nrm = xor_add(nrm, 1);
            nrm = xor_add(nrm, 8);
            nrm = xor_add(nrm, 16);
            nrm = __shfl_sync(0xffffffffu, nrm, 0);
            if (lane < kCtas) remote_store(remote_addr(part + gw, lane), nrm);
        }
        __syncwarp();
        cluster_wait();
        // stage 2: 1 -> 0
        if (element_warp) {
            const double k = rhs(buf + 2 * sz, buf + 3 * sz);
            z = __fma_rn(dt3, k, z);
            cur = __fma_rn(dt2, k, y);
        }
        publish(0);
        cluster_wait();
        // stage 3: 0 -> 1
        if (element_warp) {
            const double k = rhs(buf, buf + sz);
            z = __fma_rn(dt3, k, z);
            cur = __fma_rn(dt, k, y);
        } else {
            double r = 0.0;
            for (int i = lane; i < kCtas * warps; i += 32) r += part[i];
            for (int o = 16; o > 0; o >>= 1) r = xor_add(r, o);
            r = scale * sqrt(r);
            int stop = 0;
            if (!(P > 0.0) || !isfinite(P) || !isfinite(r)) stop = kCtlNonFinite;
            else if (r < tol) stop = kCtlConverged;
            else if (step >= max_steps) stop = kCtlMaxSteps;
            if (lane == 0) {
                if (stop) s_stop = stop;
                if (cta == 0) {
                    ctl->resid = r;
                    ctl->resid_step = step;
                }
            }
        }
        publish(1);
        cluster_wait();
        if (s_stop) {
            stopped = true;
            break;
        }
        // stage 4: 1 -> 0
        if (element_warp) {
            const double k = rhs(buf + 2 * sz, buf + 3 * sz);
            y = s_scale * __fma_rn(dt6, k, z);
            cur = y;
        }
        publish(0);
        cluster_wait();
        ++step;
        if (++ran >= limit) break;
    }
    if (own && l < 2) {
        w.y[(even ? 0 : plane) + (size_t)a * np + b] = y;
        if (!diag) w.y[(even ? 0 : plane) + (size_t)b * np + a] = even ? y : -y;
    }
    if (cta == 0 && tid == 0) {
        ctl->step = step;
        ctl->scale = s_scale;
        ctl->trace = s_trace;
        if (stopped) {
            ctl->status = s_stop;
            ctl->done = 1;
        }
    }
}

int element_warps(int n) { return (n * (n + 1) / 2 + kCtas * kOctets - 1) / (kCtas * kOctets); }

int small_smem(int n, int nnz) {
    return (5 * n * small_ld(n) + nnz + kCtas * element_warps(n)) * (int)sizeof(double) +
           (n + 1 + nnz) * (int)sizeof(int);
}

static_assert(kSmallMaxN * (kSmallMaxN + 1) / 2 <= 31 * kCtas * kOctets, "an octet per element in 31 warps per CTA");

}  // namespace

cudaError_t init_small(int n, int nnz) { return raise_smem_limit_t(small_rk4_kernel, small_smem(n, nnz)); }

cudaError_t launch_small_rk4(const DevOps &ops, const Work &w, int nnz, int limit, cudaStream_t s) {
    const int warps = element_warps(ops.n);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kCtas);
    cfg.blockDim = dim3(32 * (warps + 1));
    cfg.dynamicSmemBytes = (size_t)small_smem(ops.n, nnz);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kCtas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, small_rk4_kernel, ops, w, warps, nnz, limit);
}

}  // namespace qpr
