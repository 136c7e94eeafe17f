// Mixed-precision RK4 with an exact FP64 reference ("delta form").
//
// f is linear, so for any reference state R and stage input Y_s
//     f(Y_s) = f(R) + f(Y_s - R).
// Every refresh (start of every block of `ref_refresh` steps) sets
// R = y / tr(y), computes F = f(R) exactly in FP64 (the sparse FP64 stage
// kernel, stage 0), and takes ||F||_F as the exact FP64 residual of that step.
// Between refreshes the stage inputs are carried as FP32 deltas
// delta_s = Y_s - R and only f(delta_s) is evaluated, in FP32:
//   stage 1: k1 = F + f(D),   S  = f(D),     da = D + dt/2 k1   (D = y - R)
//   stage 2: k2 = F + f(da),  S += 2 f(da),  db = D + dt/2 k2
//   stage 3: k3 = F + f(db),  S += 2 f(db),  da = D + dt k3
//   stage 4: k4 = F + f(da),  y += dt F + dt/6 (S + f(da)) in FP64,  D = y - R
// (the weights sum to 6, so the F part of the RK4 sum is added once, in FP64)
// FP64 is used for the RK accumulation into y, the trace renormalisation and
// the exact residual; everything else runs on the FP32 pipe (GB300 has
// roughly 1/64 of its FP32 rate in FP64). The error of an FP32 f(delta) is
// relative to |H| |delta|, and |delta| shrinks with the residual, so the
// steady state reached is the FP64 one (the final answer is always
// re-checked with an exact FP64 residual).
//
// The stage kernel forms X = H delta from the CSR of H in FP32 (one warp per
// row, four nonzeros per warp instruction, float4 per lane, fixed-order
// reduction) and fuses the Lindblad right-hand side and the stage update
// into the epilogue, writing tile (I, J) and its conjugate transpose.
#include <math.h>

#include "mixed_body.cuh"

namespace qpr {
namespace {

using namespace mixed;

template <int STAGE>
__global__ void __launch_bounds__(NT)
stage_mixed_sparse_kernel(DevOps ops, MixedWork w) {
    extern __shared__ __align__(16) uint8_t dyn_smem[];
    __shared__ int s_done;
    if (threadIdx.x == 0) s_done = *(volatile int *)&w.ctl->done;
    __syncthreads();
    if (s_done) return;
    mixed_sparse_tile<STAGE>(ops, w, w.pairs[blockIdx.x].x, w.pairs[blockIdx.x].y, blockIdx.x, blockIdx.x == 0,
                             dyn_smem);
}

template <int STAGE>
cudaError_t set_mixed_attr() {
    return cudaFuncSetAttribute(stage_mixed_sparse_kernel<STAGE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kMixedDynSmem);
}

__global__ void __launch_bounds__(256) refresh_trace_kernel(DevOps ops, MixedWork w) {
    __shared__ int s_done;
    if (threadIdx.x == 0) s_done = *(volatile int *)&w.ctl->done;
    __syncthreads();
    if (s_done) return;
    refresh_trace_body(ops, w);
}

__global__ void refresh_normalize_kernel(DevOps ops, MixedWork w) {
    if (*(volatile int *)&w.ctl->done) return;  // set before this kernel started, uniform
    refresh_normalize_body(ops, w, blockIdx.x * (size_t)blockDim.x + threadIdx.x, (size_t)gridDim.x * blockDim.x);
}

__global__ void __launch_bounds__(256) refresh_post_kernel(DevOps ops, MixedWork w) {
    __shared__ int s_done;
    if (threadIdx.x == 0) s_done = *(volatile int *)&w.ctl->done;
    __syncthreads();
    if (s_done) return;
    refresh_post_body(ops, w, blockIdx.x * (size_t)blockDim.x + threadIdx.x, (size_t)gridDim.x * blockDim.x,
                      blockIdx.x == 0);
}

int grid_elems(size_t work) {
    size_t b = (work + 255) / 256;
    if (b > 152 * 8) b = 152 * 8;
    return (int)(b < 1 ? 1 : b);
}

}  // namespace

cudaError_t init_stage_mixed() {
    cudaError_t e = set_mixed_attr<1>();
    if (e == cudaSuccess) e = set_mixed_attr<2>();
    if (e == cudaSuccess) e = set_mixed_attr<3>();
    if (e == cudaSuccess) e = set_mixed_attr<4>();
    return e;
}

void launch_mixed_refresh(const DevOps &ops, const MixedWork &w, cudaStream_t s) {
    const size_t tot = 2 * (size_t)ops.np * ops.np;
    refresh_trace_kernel<<<1, 256, 0, s>>>(ops, w);
    refresh_normalize_kernel<<<grid_elems(tot), 256, 0, s>>>(ops, w);
    // F = f(R) in FP64 (stage 0: reads w.y, writes w.z): the sparse stage
    // kernel, or with a dense H the digit products (N = 900, unit weights: the
    // sparse kernel's 394 gathers a row made a refresh 1750 us; now 180)
    Work w64{};
    w64.y = w.R;
    w64.z = w.F;
    w64.ya = w.R;
    w64.yb = w.R;
    w64.g = w.g64;
    w64.partials = w.partials;
    w64.pairs = w.pairs;
    w64.pairs64 = w.pairs64;
    w64.npairs = w.npairs;
    w64.tiles = w.tiles;
    w64.ctl = w.ctl;
    if (w.digits) {
        launch_stage_digits(0, ops, w64, *w.digits, *w.digitmaps, s);
    } else {
        launch_stage_sparse(0, ops, w64, s);
    }
    refresh_post_kernel<<<grid_elems(tot), 256, 0, s>>>(ops, w);
}

void launch_mixed_stage(int stage, const DevOps &ops, const MixedWork &w, cudaStream_t s, int parts, bool serial) {
    if (w.cmaps) {  // column-block form: parts 1 = SpMM (with the gain beside it), 2 = epilogue, 4 = gain (serial)
        launch_cols_stage(stage, ops, w, s, parts, serial);
        return;
    }
    if (w.splitD) {  // dense form: the same two launches
        if (parts & 1) launch_mixed_tc_product(stage, ops, w, *w.maps, s, !serial);
        if (parts & 2) launch_x_epilogue(stage, ops, w, s, !serial);
        return;
    }
    // the sparse stage kernel computes the gain and the stop decision itself
    if (parts & 2) {
        switch (stage) {
            case 1: stage_mixed_sparse_kernel<1><<<w.npairs, NT, kMixedDynSmem, s>>>(ops, w); break;
            case 2: stage_mixed_sparse_kernel<2><<<w.npairs, NT, kMixedDynSmem, s>>>(ops, w); break;
            case 3: stage_mixed_sparse_kernel<3><<<w.npairs, NT, kMixedDynSmem, s>>>(ops, w); break;
            default: stage_mixed_sparse_kernel<4><<<w.npairs, NT, kMixedDynSmem, s>>>(ops, w); break;
        }
    }
}

}  // namespace qpr
