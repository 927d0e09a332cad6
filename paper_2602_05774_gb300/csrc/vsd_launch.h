// vsd_launch.h -- host-side launchers of the VSD kernels, one set per logit
// dtype (defined in vsd_kernels_f32.cu and vsd_kernels_bf16.cu).
#pragma once

#include <cuda_runtime.h>

#include "vsd_passes.cuh"
#include "vsd_tree.cuh"

namespace vsd {

template <typename T> struct Launch {
    // z~ ~ q per row, tokens/logq/row_stats written from the row records
    static cudaError_t sample(const Problem<T>& P, bool vec, cudaStream_t s);
    // verification of given tokens (linear paths): rows, accepted lengths, residual
    // draws, corrected paths, log-kappa
    static cudaError_t verify(const Problem<T>& P, bool vec, cudaStream_t s);
    // the same in one kernel, for few rows
    static cudaError_t verify_few(const Problem<T>& P, bool vec, cudaStream_t s);
    // log kappa of supplied greedy reference paths: [B][D] rows -> out [B][D]
    static cudaError_t reference(const Problem<T>& P, bool vec, float* out, cudaStream_t s);
    // tree verification, each branch alone: node rows; then per row the residual
    // draws, per tree the nodes' outputs and the bonus
    static cudaError_t tree(const Problem<T>& P, bool vec, cudaStream_t s);
    // tree verification with the sequential sibling rule
    static cudaError_t tree_seq(const Problem<T>& P, bool vec, cudaStream_t s);
    // the E-step + M-step over draft trees (node rows, per-tree M-step, gradient rows)
    static cudaError_t tree_em(const Problem<T>& P, bool vec, const vsd_tree_em_outputs& o,
                               void* grad, bool grad_bf16, cudaStream_t s);
    // M-step weights and loss from an E-step view
    static cudaError_t weights(const Problem<T>& P, const EStepView& E, float* weights,
                              float* loss, cudaStream_t s);
    // gradient rows from coefficients and row statistics
    static cudaError_t grad(const Problem<T>& P, bool vec, const float4* rstats, void* grad,
                            bool grad_bf16, cudaStream_t s);
    // the fused persistent E-step + M-step kernel
    static cudaError_t fused(const Problem<T>& P, bool vec, void* grad, bool grad_bf16,
                             int ctas, cudaStream_t s);
    // the E-step + M-step in two kernels (rows with paths and M-steps; gradient)
    static cudaError_t staged(const Problem<T>& P, bool vec, void* grad, bool grad_bf16,
                              cudaStream_t s);
    // the gradient rows from the records and coefficients that an E-step + M-step
    // left in the workspace (a programmatic dependent launch)
    static cudaError_t grad_rows(const Problem<T>& P, bool vec, void* grad, bool grad_bf16,
                                 cudaStream_t s);
    // resident blocks per SM of the fused kernel
    static int fused_blocks_per_sm(const Problem<T>& P, bool vec, bool grad_bf16);
};

// Host-side per-device caches, so that a call makes no attribute or
// occupancy query once a kernel has been set up on its device (vsd_api.cu).
// The SM count of the current device.
int device_sm_count();
// Lets `kernel` use `smem` bytes of dynamic shared memory on the current
// device (cudaFuncSetAttribute only when a larger size than before is asked).
cudaError_t ensure_dyn_smem(const void* kernel, size_t smem);
// Resident blocks per SM of `kernel` with `threads` threads and `smem` bytes
// of dynamic shared memory on the current device (0 on error).
int blocks_per_sm(const void* kernel, int threads, size_t smem);

inline size_t table_smem_bytes(int nch) { return (size_t)nch * sizeof(float4); }
// Dynamic shared memory of a streaming kernel: the TMA ring of S stages (vector
// rows only; at least MIN bytes) followed by the chunk table.
template <int S, size_t MIN = 0> inline size_t stream_smem_bytes(int nch, bool vec) {
    return (vec ? ring_bytes<S, MIN>() : 0) + table_smem_bytes(nch);
}

// Whether a kernel of one block per row takes the ring of kDeepStages: rows of
// at least 48 chunks (96 KB), all of them resident at per_sm blocks per SM, so
// that each row's own stream bounds the call.  us, one stage / two stages:
//   verification, float32: V=65536 R=304 83 / 68, V=128256 R=304 141 / 113, R=608
//     185 / 167; bf16: V=128256 R=304 87 / 74, R=608 107 / 102, R=4096 396 / 402
//   E-step + M-step without a gradient, V=128256: float32 R=304 143 / 115, R=608
//     180 / 172; bf16 R=304 88 / 80, R=608 111 / 119 (per_sm = 2)
//   reference rows, bf16: V=128256 R=304 50 / 44, R=512 66 / 66; V=524288 R=304
//     136 / 120, R=512 185 / 204 (per_sm = 2 from 256 chunks on)
//   trees of 8 nodes, float32, V=128256 R=304: alone 130 / 101, sequential rule
//     243 / 214, E-step + M-step 207 / 184
inline bool deep_ring(bool vec, int nch, int64_t rows, int per_sm = 4) {
    return vec && nch >= 48 && rows <= per_sm * (int64_t)device_sm_count();
}
// That kernel's instance (deep, vec: names in the launcher; the further template
// arguments, each with a comma before it).
#define VSD_BY_RING(kern, T_, ...)                                   \
    (deep ? kern<T_, true __VA_ARGS__, kDeepStages>                  \
          : vec ? kern<T_, true __VA_ARGS__, kRowStages> : kern<T_, false __VA_ARGS__, kRowStages>)
template <size_t MIN = 0> inline size_t row_smem_bytes(int nch, bool vec, bool deep) {
    return deep ? stream_smem_bytes<kDeepStages, MIN>(nch, vec)
                : stream_smem_bytes<kRowStages, MIN>(nch, vec);
}

// The draft LM head on the tensor cores (vsd_lmhead.cu): logits = hidden .
// weight^T, bf16 in, fp32 accumulation, bf16 out; status collects timeouts.
bool lmhead_shape_ok(const void* hidden, const void* weight, const void* logits, int M, int N,
                     int K);
// With chunk_tab, the epilogue also writes chunk_tab[r * chunk_stride + ch].xy
// = (max, sum 2^{(x - max) chunk_c}) of row r's bf16 logits x in columns
// [1024 ch, 1024 ch + 1024): the draft half of the E-step's chunk table.
cudaError_t lmhead_gemm(const void* hidden, const void* weight, int M, int N, int K, void* logits,
                        int* status, uint64_t timeout_ns, cudaStream_t s,
                        float4* chunk_tab = nullptr, int chunk_stride = 0, float chunk_c = 0.f);
// The LM head's backward (vsd_lmhead_bwd.cu): d_hidden = G . weight and
// d_weight = G^T . hidden (fp32, either may be null), with G the gradient of
// the bf16 draft logits made on chip from the E-step's row records, M-step
// coefficients and (klr non-null) top-K terms.
// fac_scratch: lmhead_backward_fac_bytes(R) bytes of device memory, 16-byte
// aligned, for the rows' packed factors.
size_t lmhead_backward_fac_bytes(int R);
cudaError_t lmhead_backward(const void* hidden, const void* weight, const void* logits, int R,
                            int V, int H, float T, const RowRec* rows, const Coef* coef,
                            const KlRec* klr, void* fac_scratch, float* d_hidden,
                            float* d_weight, int* status, uint64_t timeout_ns, cudaStream_t s);
// The same products from G itself, bf16 [R][V].
cudaError_t lmhead_backward_dense(const void* hidden, const void* weight, const void* G, int R,
                                  int V, int H, float* d_hidden, float* d_weight, int* status,
                                  uint64_t timeout_ns, cudaStream_t s);

}  // namespace vsd
