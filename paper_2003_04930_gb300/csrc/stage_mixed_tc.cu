// Dense mixed-form RK4 stage on the 5th-generation tensor cores (tcgen05).
//
// X = H delta for an FP32 stage delta is formed as a 3-term split-BF16
// product with FP32 accumulation: H = H0 + H1 + H2 and delta = d0 + d1 + d2
// (each term the BF16 rounding of what the previous terms left), and
//     X = sum over i + j <= 2 of H_i d_j
// (the dropped terms are below 2^-24 relative). Planes of H that are zero are
// left out: three products instead of six where BF16 holds every entry, as
// with unit weights. Because delta is Hermitian the B operand of columns J is
// K-major with rows [Re delta_J ; -Im delta_J], so the product is one GEMM
// [Re X | Im X] = H [Re delta | Im delta].
//
// mixed_gemm_kernel is persistent: one CTA per SM takes 128 x 128 tiles of
// [Re X | Im X]. Warp 0 (one thread) streams, per K block of 64, the planes
// of H and the three of delta with TMA (128-byte swizzle); warp 1 (one
// thread) issues every product of the block from them, so each plane is read
// once for all its products; warps 4 to 7 write the tile before from the
// other half of TMEM meanwhile. The small products (i + j >= 1) and the
// dominant H0 d0 accumulate separately and are added once, in FP32: the
// tensor core's accumulation does not round to nearest, so its error grows
// with every K step added to a large accumulator. The grid's first CTAs form
// the gain (and, at stage 2, the stop decision). The Lindblad right-hand
// side and the RK4 update are the column forms' epilogue (stage_cols.cu),
// which also writes the BF16 split of the next stage input.
//
// Why a product kernel of its own: with the epilogue in the product kernel a
// CTA owned a pair of 128 x 128 complex tiles, 36 of them at N = 900 on 152
// SMs, and no tensor instruction ran during its epilogue: 115 us a stage and
// 12 for the gain at N = 900 with unit weights; now 27 us a stage, 17 of them
// this kernel.
//
// Every mbarrier wait gives up after a bounded time, sets ctl->err_timeout
// and ends the CTA's work; TMEM is always released.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>
#include <math.h>

#include <algorithm>

#include "cols_body.cuh"
#include "cols_spmm.cuh"
#include "mixed_body.cuh"
#include "qpr_internal.cuh"
#include "tma_util.cuh"

namespace qpr {
namespace {

constexpr int TB = kTileTc;             // 128: rows of a tile and its columns of one plane
constexpr int BK = 64;                  // BF16 K per stage: one 128-byte swizzle row
constexpr int OP_BYTES = TB * BK * 2;   // 16 KB: one plane's operand tile
constexpr int NTHREADS = 256;
constexpr int kRingBytes = 192 * 1024;
constexpr int kMaxStages = 3;
constexpr int LDT = 33;                 // staged output row: 32 values
constexpr int STORE_BYTES = 4 * 32 * LDT * 4;  // one 32 x 32 block per storing warp
constexpr int SMEM_BYTES = kRingBytes + STORE_BYTES + 1024;  // + alignment slack
constexpr uint32_t TMEM_COLS = 512;     // two buffers of (128 dominant, 128 small)

static_assert(SMEM_BYTES <= 227 * 1024, "shared memory");

using tma::mbar_expect_tx;
using tma::mbar_init;
using tma::mbar_wait;
using tma::smem_u32;
using tma::load_3d;
using tma::load_4d;

// Shared-memory matrix descriptor: K-major operand in the canonical 128-byte
// swizzled layout written by TMA (8 rows x 128 B atoms, 1024 B between
// 8-row groups).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);          // start address
    d |= (uint64_t)1 << 16;                          // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)((1024 >> 4) & 0x3FFF) << 32;     // stride byte offset: 8 rows x 128 B
    d |= (uint64_t)1 << 46;                          // descriptor version
    d |= (uint64_t)2 << 61;                          // 128-byte swizzle
    return d;
}

// Instruction descriptor, kind::f16: BF16 A and B (K-major), FP32 D, M = 128, N = 128.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TB >> 3) << 17) |
                            ((uint32_t)(128 >> 4) << 24);

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(accumulate));
}
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                     smem_u32(bar))
                 : "memory");
}
// 32 columns of this warp's TMEM lanes, dominant and small parts together.
__device__ __forceinline__ void tmem_ld32x2(uint32_t tb, uint32_t ts, uint32_t (&r)[32], uint32_t (&q)[32]) {
#define QPR_LD32(v, addr)                                                                                              \
    asm volatile(                                                                                                      \
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"  \
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"                                              \
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),              \
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),        \
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),      \
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])       \
        : "r"(addr))
    QPR_LD32(r, tb);
    QPR_LD32(q, ts);
#undef QPR_LD32
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; i += 8)
#pragma unroll
        for (int k = 0; k < 8; ++k) asm volatile("" : "+r"(r[i + k]), "+r"(q[i + k]));
}

// levels: planes of H that are not zero (1 to 3); stages: depth of the ring;
// tiles of the product; ng: leading CTAs that form the gain.
template <int STAGE>
__global__ void __launch_bounds__(NTHREADS, 1)
mixed_gemm_kernel(DevOps ops, MixedWork w, const __grid_constant__ CUtensorMap tmH,
                  const __grid_constant__ CUtensorMap tmIn, int levels, int stages, int ng) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base_sh;
    __shared__ int s_done, s_fail;
    if ((int)blockIdx.x < ng) {
        cols::gain_role<STAGE == 2>(ops, w, blockIdx.x, ng, [&] { return w.pv; });
        return;
    }
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    Ctl *ctl = w.ctl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int np = ops.np, T = np / TB, nkb = np / BK;
    const int tiles = 2 * T * T, step = gridDim.x - ng, first = blockIdx.x - ng;
    const int stage_bytes = (levels + 3) * OP_BYTES;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_base_sh)),
                     "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    if (tid == 32) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4);
        }
        tma::mbar_init_fence();
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_base_sh;
    tma::grid_dependency_wait();
    tma::launch_dependents();
    if (tid == 0) {
        s_done = *(volatile int *)&ctl->done;
        s_fail = 0;
    }
    __syncthreads();

    if (s_done) {
    } else if (warp == 0 && lane == 0) {
        // TMA producer: tile t is rows (t % T) of H, columns t / T (plane, then column tile)
        bool ok = true;
        int it = 0;
        for (int t = first; t < tiles && ok; t += step) {
            const int rt = t % T, ct = t / T, pl = ct / T, jt = ct - pl * T;
            for (int kb = 0; kb < nkb; ++kb, ++it) {
                const int st = it % stages;
                if (it >= stages && !mbar_wait(&empty_bar[st], ((it / stages) - 1) & 1)) {
                    ok = false;
                    break;
                }
                uint8_t *sb = smem + st * stage_bytes;
                mbar_expect_tx(&full_bar[st], (uint32_t)stage_bytes);
                for (int i = 0; i < levels; ++i) load_3d(sb + i * OP_BYTES, &tmH, &full_bar[st], kb * BK, rt * TB, i);
                for (int j = 0; j < 3; ++j)
                    load_4d(sb + (levels + j) * OP_BYTES, &tmIn, &full_bar[st], kb * BK, jt * TB, pl, j);
            }
        }
        if (!ok) atomicExch(&s_fail, 1);
    } else if (warp == 1 && lane == 0) {
        // MMA issuer
        bool ok = true;
        int it = 0, n = 0;
        for (int t = first; t < tiles && ok; t += step, ++n) {
            const int buf = n & 1;
            if (n >= 2) ok = mbar_wait(&acc_empty[buf], ((n >> 1) - 1) & 1);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t big = tmem + (uint32_t)(buf * 2 * TB), small = big + TB;
            for (int kb = 0; kb < nkb; ++kb, ++it) {
                const int st = it % stages;
                if (!mbar_wait(&full_bar[st], (it / stages) & 1)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t sa = smem_u32(smem + st * stage_bytes), sb = sa + levels * OP_BYTES;
                bool fresh = kb == 0;
                // (0,2) (1,1) (2,0) (0,1) (1,0), smallest first, then (0,0)
                for (int d = 2; d >= 0; --d)
                    for (int i = 0; i <= d && i < levels; ++i) {
                        const uint64_t dA = sw128_desc(sa + i * OP_BYTES), dB = sw128_desc(sb + (d - i) * OP_BYTES);
                        const uint32_t dst = d ? small : big;
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
                            const uint64_t adv = (uint64_t)((kk * 32) >> 4);  // 16 BF16 = 32 bytes along K
                            umma_bf16(dst, dA + adv, dB + adv, (kk > 0 || !(d ? fresh : kb == 0)) ? 1u : 0u);
                        }
                        if (d) fresh = false;
                    }
                umma_commit(&empty_bar[st]);
            }
            umma_commit(&acc_full[buf]);
        }
        if (!ok) atomicExch(&s_fail, 1);
    } else if (warp >= 4) {
        // the tile before: 32 rows per warp, 32 columns at a time through shared memory
        const int q = warp & 3;
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        float *sT = reinterpret_cast<float *>(smem + kRingBytes) + q * 32 * LDT;
        const size_t plane = (size_t)np * np;
        int n = 0;
        for (int t = first; t < tiles; t += step, ++n) {
            const int buf = n & 1;
            const int rt = t % T, ct = t / T, pl = ct / T, jt = ct - pl * T;
            const bool ok = mbar_wait(&acc_full[buf], (n >> 1) & 1);
            if (__any_sync(0xffffffffu, !ok)) {
                if (lane == 0) atomicExch(&s_fail, 1);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            float *out = w.X + pl * plane + (size_t)(rt * TB + q * 32) * np + jt * TB;
            for (int c = 0; c < TB; c += 32) {
                uint32_t vb[32], vs[32];
                const uint32_t base = tmem + lane_off + (uint32_t)(buf * 2 * TB + c);
                tmem_ld32x2(base, base + TB, vb, vs);
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 32; ++i) sT[lane * LDT + i] = __fadd_rn(__uint_as_float(vb[i]), __uint_as_float(vs[i]));
                __syncwarp();
#pragma unroll 8
                for (int r = 0; r < 32; ++r) out[(size_t)r * np + c + lane] = sT[r * LDT + lane];
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&acc_empty[buf])) : "memory");
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (tid == 0 && s_fail) atomicExch(&ctl->err_timeout, 1);
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TMEM_COLS));
    }
}

template <int STAGE>
cudaError_t set_attr() {
    return cudaFuncSetAttribute(mixed_gemm_kernel<STAGE>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode_impl() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void *p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

}  // namespace

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() { return get_encode_impl(); }

cudaError_t init_mixed_tc() {
    cudaError_t e = set_attr<1>();
    if (e == cudaSuccess) e = set_attr<2>();
    if (e == cudaSuccess) e = set_attr<3>();
    if (e == cudaSuccess) e = set_attr<4>();
    return e;
}

// Tensor maps: H planes [3][np][np] and delta-split planes [3][2][np][np],
// BF16, boxes of 64 (K) x 128 rows, 128-byte swizzle.
bool make_tc_maps(const DevOps &ops, const __nv_bfloat16 *hsplit, int levels, int sms,
                  const __nv_bfloat16 *const dsplit[3], TcMaps *maps) {
    maps->levels = levels;
    maps->sms = sms;
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t np = (cuuint64_t)ops.np;
    {
        cuuint64_t dims[3] = {np, np, 3};
        cuuint64_t strides[2] = {np * 2, np * np * 2};
        cuuint32_t box[3] = {BK, TB, 1};
        cuuint32_t es[3] = {1, 1, 1};
        if (enc(&maps->h, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void *)hsplit, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    for (int i = 0; i < 3; ++i) {
        cuuint64_t dims[4] = {np, np, 2, 3};
        cuuint64_t strides[3] = {np * 2, np * np * 2, 2 * np * np * 2};
        cuuint32_t box[4] = {BK, TB, 1, 1};
        cuuint32_t es[4] = {1, 1, 1, 1};
        if (enc(&maps->d[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void *)dsplit[i], dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    return true;
}

// Stage input split planes: stage 1 D (map 0), stage 2 da (map 1), stage 3
// db (map 2), stage 4 da (map 1).
void launch_mixed_tc_product(int stage, const DevOps &ops, const MixedWork &w, const TcMaps &m, cudaStream_t s, bool pdl) {
    const int T = ops.np / TB, tiles = 2 * T * T;
    const int ng = std::min(64, std::max(8, m.sms - tiles));
    const int stages = std::min(kMaxStages, kRingBytes / ((m.levels + 3) * OP_BYTES));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ng + std::min(tiles, m.sms));
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    switch (stage) {
        case 1: cudaLaunchKernelEx(&cfg, mixed_gemm_kernel<1>, ops, w, m.h, m.d[0], m.levels, stages, ng); break;
        case 2: cudaLaunchKernelEx(&cfg, mixed_gemm_kernel<2>, ops, w, m.h, m.d[1], m.levels, stages, ng); break;
        case 3: cudaLaunchKernelEx(&cfg, mixed_gemm_kernel<3>, ops, w, m.h, m.d[2], m.levels, stages, ng); break;
        default: cudaLaunchKernelEx(&cfg, mixed_gemm_kernel<4>, ops, w, m.h, m.d[1], m.levels, stages, ng); break;
    }
}

}  // namespace qpr
