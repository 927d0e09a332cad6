// vsd_lmhead.cu -- the draft model's LM head on the tensor cores:
// logits[M][N] = hidden[M][K] . weight[N][K]^T, bf16 inputs, fp32 accumulation
// in tensor memory (TMEM), bf16 logits out (the draft head that produces q,
// paper Sec. 5 implementation details), and, for the E-step + M-step that
// follows (vsd_lmhead_estep_mstep), each row's chunk statistics.  The GEMM is
// vsd_gemm2.cuh's on CTA pairs, both operands K-major as they lie; logits of up
// to 128 rows alone are made by k_logits_few below.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <mutex>

#include "vsd.h"
#include "vsd_gemm2.cuh"
#include "vsd_launch.h"

namespace vsd_lm {

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// against the driver library).
EncodeTiledFn encode_fn() {
    static std::once_flag once;
    static EncodeTiledFn fn = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// Tensor map of a row-major bf16 matrix [rows][cols] read in boxes of box_rows x
// box_cols, swizzled in swizzle_bytes; out-of-range elements read as zero (they
// add nothing to a dot product).
bool make_map_box(CUtensorMap* m, const void* base, int rows, int cols, int box_cols,
                  int box_rows, int swizzle_bytes) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
               box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               swizzle_bytes == 128  ? CU_TENSOR_MAP_SWIZZLE_128B
               : swizzle_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                     : CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

// ---------------------------------------------------------------- few rows
// Logits of M <= 128 rows, one CTA per 128 x 256 tile: the weight's stream bounds
// these calls, and a pair, whose second CTA would hold rows beyond M, keeps 96 KB
// of it per SM in flight where this keeps 128.  With fewer tiles than pairs both
// SMs of a pair stream one tile, which is faster unless K is small, where a pair's
// start and end cost more.  us, M = 64, here / on pairs: N = 128256 K = 4096 190 /
// 194, K = 256 26 / 32; N = 32000 K = 4096 63 / 69; N = 8000 K = 4096 38 / 34; N =
// 256 K = 256 9 / 13.
//   warp 0     TMA producer, 4 stages;
//   warp 1     MMA issuer: tcgen05.mma M = 128, N = 256, K = 16 into one of two
//              accumulators;
//   warps 2-5  epilogue: each its 32 rows, rounded to bf16.
// Waits are bounded as in vsd_gemm2.cuh, and the CTA leaves when the arrivals of
// its copies and commits have landed.
constexpr int kFewRows = 128, kFewN = 256, kFewK = 64, kFewStages = 4, kFewThreads = 192;
constexpr int kFewA = kFewRows * kFewK * 2, kFewStage = kFewA + kFewN * kFewK * 2;
struct FewBars {
    uint64_t full[kFewStages], empty[kFewStages];
    uint64_t acc_full[2], acc_empty[2], drain;
    uint32_t tmem_base;
    int err;
};
constexpr size_t kFewSmem = 1024 + kFewStages * kFewStage + sizeof(FewBars);

__global__ void __launch_bounds__(kFewThreads, 1)
    k_logits_few(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 __nv_bfloat16* __restrict__ out, int M, int N, int K, int* status,
                 uint64_t timeout_ns) {
    extern __shared__ unsigned char dsm_raw[];
    unsigned char* dsm = dsm_raw + ((1024u - (smem_u32(dsm_raw) & 1023u)) & 1023u);
    FewBars* sb = reinterpret_cast<FewBars*>(dsm + kFewStages * kFewStage);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntiles = (N + kFewN - 1) / kFewN, nk = (K + kFewK - 1) / kFewK;
    constexpr uint32_t kIdesc = idesc_bf16(kFewRows, kFewN);
    if (threadIdx.x == 0) {
        for (int s = 0; s < kFewStages; ++s) {
            mbar_init(&sb->full[s], 1);
            mbar_init(&sb->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sb->acc_full[b], 1);
            mbar_init(&sb->acc_empty[b], 4);
        }
        mbar_init(&sb->drain, 1);
        sb->err = 0;
        mbar_init_fence();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&sb->tmem_base)), "r"(2 * kFewN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sb->tmem_base;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
        return wait_phase_err(bar, parity, &sb->err, timeout_ns, status);
    };
    if (warp == 0) {
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int t = blockIdx.x; ok && t < ntiles && !*(volatile int*)&sb->err; t += gridDim.x)
                for (int kb = 0; kb < nk; ++kb, ++it) {
                    const int s = (int)(it % kFewStages);
                    const uint32_t round = it / kFewStages;
                    if (round > 0 && !wait(&sb->empty[s], (round - 1) & 1u)) {
                        ok = false;
                        break;
                    }
                    unsigned char* a = dsm + s * kFewStage;
                    mbar_expect_tx(&sb->full[s], kFewStage);
                    tma_load_2d(a, &tmA, kb * kFewK, 0, &sb->full[s]);
                    tma_load_2d(a + kFewA, &tmB, kb * kFewK, t * kFewN, &sb->full[s]);
                }
            for (uint32_t j = it > (uint32_t)kFewStages ? it - kFewStages : 0; j < it; ++j)
                wait_phase_drain(&sb->full[j % kFewStages], (j / kFewStages) & 1u, timeout_ns);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            uint32_t it = 0, lt = 0;
            bool ok = true;
            for (int t = blockIdx.x; ok && t < ntiles && !*(volatile int*)&sb->err;
                 t += gridDim.x) {
                const uint32_t buf = lt & 1u, use = lt >> 1;
                if (use > 0 && !wait(&sb->acc_empty[buf], (use - 1) & 1u)) break;
                tc_fence_after();
                for (int kb = 0; kb < nk; ++kb) {
                    const int s = (int)(it % kFewStages);
                    if (!wait(&sb->full[s], (it / kFewStages) & 1u)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a = smem_u32(dsm + s * kFewStage), b = a + kFewA;
#pragma unroll
                    for (int k = 0; k < kFewK / 16; ++k)
                        mma_bf16(tmem + buf * kFewN, sdesc_sw128(a + 32u * k),
                                 sdesc_sw128(b + 32u * k), kIdesc, (kb | k) != 0 ? 1u : 0u);
                    mma_commit(&sb->empty[s]);
                    ++it;
                }
                if (!ok) break;
                mma_commit(&sb->acc_full[buf]);
                ++lt;
            }
            mma_commit(&sb->drain);
            wait_phase_drain(&sb->drain, 0, timeout_ns);
            for (uint32_t j = it > (uint32_t)kFewStages ? it - kFewStages : 0; j < it; ++j)
                wait_phase_drain(&sb->empty[j % kFewStages], (j / kFewStages) & 1u, timeout_ns);
            for (uint32_t j = lt > 2u ? lt - 2u : 0; j < lt; ++j)
                wait_phase_drain(&sb->acc_full[j & 1u], (j >> 1) & 1u, timeout_ns);
        }
    } else {
        const int q = warp & 3;  // TMEM lanes 32q .. 32q + 31
        const int row = 32 * q + lane;
        uint32_t lt = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++lt) {
            const uint32_t buf = lt & 1u;
            // (one outcome for the whole warp)
            if (!__all_sync(0xffffffffu, wait(&sb->acc_full[buf], (lt >> 1) & 1u))) break;
            tc_fence_after();
            const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16) + buf * kFewN;
#pragma unroll 1
            for (int c = 0; c < kFewN / 32; ++c) {
                uint32_t r[32];
                __syncwarp();
                tmem_ld32(taddr + 32u * c, r);
                const int col = t * kFewN + 32 * c;
                if (row >= M || col >= N) continue;
                __nv_bfloat16* o = out + (size_t)row * N + col;
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    if (col + 8 * v < N)
                        *reinterpret_cast<uint4*>(o + 8 * v) = make_uint4(
                            pack_bf16(r[8 * v], r[8 * v + 1]), pack_bf16(r[8 * v + 2], r[8 * v + 3]),
                            pack_bf16(r[8 * v + 4], r[8 * v + 5]),
                            pack_bf16(r[8 * v + 6], r[8 * v + 7]));
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sb->acc_empty[buf]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     :: "r"(tmem), "r"(2 * kFewN) : "memory");
    }
}

bool make_map_store(CUtensorMap* m, float* base, int rows, int cols, int box) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 4};
    const cuuint32_t boxes[2] = {(cuuint32_t)box, (cuuint32_t)box};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, boxes, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace vsd_lm

namespace vsd {

bool lmhead_shape_ok(const void* hidden, const void* weight, const void* logits, int M, int N,
                     int K) {
    if (!hidden || !weight || !logits) return false;
    if (M < 1 || N < 8 || K < 8) return false;
    if (N % 8 || K % 8) return false;  // 16-byte rows for TMA and for the stores
    if (((uintptr_t)hidden | (uintptr_t)weight | (uintptr_t)logits) & 15) return false;
    return true;
}

cudaError_t lmhead_gemm(const void* hidden, const void* weight, int M, int N, int K, void* logits,
                        int* status, uint64_t timeout_ns, cudaStream_t s, float4* chunk_tab,
                        int chunk_stride, float chunk_c) {
    CUtensorMap ta, tb;
    const int pairs = device_sm_count() / 2;
    if (!chunk_tab && M <= vsd_lm::kFewRows &&
        (K <= 1024 || (N + vsd_lm::kFewN - 1) / vsd_lm::kFewN > pairs)) {
        using namespace vsd_lm;
        if (!make_map_box(&ta, hidden, M, K, kFewK, kFewRows, 128) ||
            !make_map_box(&tb, weight, N, K, kFewK, kFewN, 128))
            return cudaErrorInvalidValue;
        const cudaError_t e = ensure_dyn_smem((const void*)k_logits_few, kFewSmem);
        if (e != cudaSuccess) return e;
        const int ntiles = (N + kFewN - 1) / kFewN, sms = device_sm_count();
        k_logits_few<<<ntiles < sms ? ntiles : sms, kFewThreads, kFewSmem, s>>>(
            ta, tb, static_cast<__nv_bfloat16*>(logits), M, N, K, status, timeout_ns);
        return cudaGetLastError();
    }
    if (!vsd_lm::make_map_box(&ta, hidden, M, K, vsd_g2::BK, vsd_g2::BM, 128) ||
        !vsd_lm::make_map_box(&tb, weight, N, K, vsd_g2::BK, vsd_g2::BH, 128))
        return cudaErrorInvalidValue;
    auto kern = vsd_g2::k_gemm2<false, false, vsd_g2::StoreLogits>;
    cudaError_t e = ensure_dyn_smem((const void*)kern, vsd_g2::smem_bytes<vsd_g2::StoreLogits>());
    if (e != cudaSuccess) return e;
    const long long nunits = vsd_g2::ChunkOrder::units(
        M, N, vsd_g2::StoreLogits::per_unit(chunk_tab != nullptr));
    const int grid = 2 * (int)(nunits < pairs ? nunits : pairs);
    const vsd_g2::StoreLogits epi{static_cast<__nv_bfloat16*>(logits), M, N, chunk_tab,
                                  chunk_stride, chunk_c};
    kern<<<grid, vsd_g2::kThreads, vsd_g2::smem_bytes<vsd_g2::StoreLogits>(), s>>>(ta, tb, M, N, K, epi, status,
                                                            timeout_ns);
    return cudaGetLastError();
}

}  // namespace vsd
