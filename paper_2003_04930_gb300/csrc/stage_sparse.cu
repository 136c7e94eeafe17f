// Sparse FP64 RK4 stage kernel: X = H Y with H in CSR (exact FP64, O(nnz N)
// work per stage), the gain and the same fused Lindblad/RK4 epilogue as the
// dense forms, one launch a stage.
//
// H of Eq. S6 has one nonzero per link (symmetrised) plus an optional
// diagonal, so H Y costs 4 nnz(H) N flops against 4 N^3 for the dense product.
// One CTA owns the tile pair (I, J): a warp takes a row a of tile I and
// gathers, for each nonzero H_ak, the 32 columns J of row k of Re Y and Im Y
// (two coalesced 256-byte loads), so X_IJ(a, b) = sum_k H_ak Y_kb is formed
// in registers, one column per lane. X_JI is formed the same way. The pairs
// run heaviest first (Work::pairs64), two CTAs per SM, so that the last ones
// to start are the lightest; the launches are programmatic dependent ones.
#include <algorithm>
#include <vector>

#include "sparse_body.cuh"
#include "tma_util.cuh"

namespace qpr {
namespace {

using namespace sparse64;

// Two CTAs per SM (16 warps keep the FP64 pipe busy; with more, all pairs of
// a middle-sized problem are resident at once and nothing evens them out).
constexpr int kLaunchSmem = 100 * 1024;
static_assert(kLaunchSmem >= SMEM_BYTES, "shared memory");

template <int STAGE>
__global__ void __launch_bounds__(NTHREADS, 2)
stage_sparse_kernel(DevOps ops, Work w) {
    extern __shared__ __align__(16) double smem[];
    __shared__ int s_done;
    const int4 p = w.pairs64[blockIdx.x];
    tma::grid_dependency_wait();
    tma::launch_dependents();
    // the pair (0, 0) may set `done` while other CTAs start: one read per CTA
    if (threadIdx.x == 0) s_done = *(volatile int *)&w.ctl->done;
    __syncthreads();
    if (s_done) return;
    tile<STAGE>(ops, w, p.x, p.y, p.z, p.z == 0, smem);
}

template <int STAGE>
cudaError_t set_attr() {
    return cudaFuncSetAttribute(stage_sparse_kernel<STAGE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kLaunchSmem);
}

template <int STAGE>
void launch_t(const DevOps &ops, const Work &w, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(w.npairs);
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = kLaunchSmem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, stage_sparse_kernel<STAGE>, ops, w);
}

}  // namespace

cudaError_t init_stage_sparse() {
    cudaError_t e = set_attr<0>();
    if (e == cudaSuccess) e = set_attr<1>();
    if (e == cudaSuccess) e = set_attr<2>();
    if (e == cudaSuccess) e = set_attr<3>();
    if (e == cudaSuccess) e = set_attr<4>();
    return e;
}

std::vector<int4> pairs_by_work(const HostOps &h, int np) {
    const int T = np / TS;
    std::vector<int64_t> nz(T, 0);
    for (int i = 0; i < (int)h.n; ++i) nz[i / TS] += h.hptr[i + 1] - h.hptr[i];
    std::vector<int4> p;
    std::vector<int64_t> work;
    for (int pass = 0; pass < 2; ++pass)
        for (int I = 0; I < T; ++I)
            for (int J = pass ? I : I + 1; J < (pass ? I + 1 : T); ++J) {
                p.push_back(make_int4(I, J, (int)p.size(), 0));
                work.push_back(I == J ? nz[I] : nz[I] + nz[J]);
            }
    std::stable_sort(p.begin(), p.end(), [&](const int4 &a, const int4 &b) { return work[a.z] > work[b.z]; });
    return p;
}

void launch_stage_sparse(int stage, const DevOps &ops, const Work &w, cudaStream_t s) {
    switch (stage) {
        case 0: launch_t<0>(ops, w, s); break;
        case 1: launch_t<1>(ops, w, s); break;
        case 2: launch_t<2>(ops, w, s); break;
        case 3: launch_t<3>(ops, w, s); break;
        default: launch_t<4>(ops, w, s); break;
    }
}

}  // namespace qpr
