// vsd_lmhead.cu -- the draft model's LM head on the tensor cores:
// logits[M][N] = hidden[M][K] . weight[N][K]^T, bf16 inputs, fp32 accumulation
// in tensor memory (TMEM), bf16 logits out (the draft head that produces q,
// paper Sec. 5 implementation details), and, for the E-step + M-step that
// follows (vsd_lmhead_estep_mstep), each row's chunk statistics.  The GEMM is
// vsd_gemm2.cuh's on CTA pairs, both operands K-major as they lie.
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

// Tensor map of a row-major bf16 matrix [rows][cols] read in boxes of
// box_rows x 64 columns with the 128-byte swizzle; out-of-range elements read
// as zero (they add nothing to a dot product).
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
    if (!vsd_lm::make_map_box(&ta, hidden, M, K, vsd_g2::BK, vsd_g2::BM, 128) ||
        !vsd_lm::make_map_box(&tb, weight, N, K, vsd_g2::BK, vsd_g2::BH, 128))
        return cudaErrorInvalidValue;
    auto kern = vsd_g2::k_gemm2<false, false, vsd_g2::StoreLogits>;
    cudaError_t e = ensure_dyn_smem((const void*)kern, vsd_g2::smem_bytes<vsd_g2::StoreLogits>());
    if (e != cudaSuccess) return e;
    const long long nunits = vsd_g2::ChunkOrder::units(
        M, N, vsd_g2::StoreLogits::per_unit(chunk_tab != nullptr));
    const int pairs = device_sm_count() / 2;
    const int grid = 2 * (int)(nunits < pairs ? nunits : pairs);
    const vsd_g2::StoreLogits epi{static_cast<__nv_bfloat16*>(logits), M, N, chunk_tab,
                                  chunk_stride, chunk_c};
    kern<<<grid, vsd_g2::kThreads, vsd_g2::smem_bytes<vsd_g2::StoreLogits>(), s>>>(ta, tb, M, N, K, epi, status,
                                                            timeout_ns);
    return cudaGetLastError();
}

}  // namespace vsd
