// vsd_staged_impl.cuh -- launchers of the two-kernel E-step + M-step for one
// logit dtype VSD_T.  Included once by vsd_staged_f32.cu and once by
// vsd_staged_bf16.cu.
#pragma once

#include "vsd_staged.cuh"

namespace vsd {

template <>
cudaError_t Launch<VSD_T>::grad_rows(const Problem<VSD_T>& P, bool vec, void* grad,
                                     bool grad_bf16, cudaStream_t s);

template <>
cudaError_t Launch<VSD_T>::staged(const Problem<VSD_T>& P, bool vec, void* grad, bool grad_bf16,
                                  cudaStream_t s) {
    // (behind the LM head the smaller block fits beside its CTAs, and streams the
    // target meanwhile)
    const bool deep =
        !P.xtab_given && deep_ring(vec, P.nch, P.R, sizeof(VSD_T) == 2 ? 2 : 4);
    const size_t smem = staged_smem_bytes(P.nch, vec, deep);
    auto rows = P.kl_topk ? VSD_BY_RING(k_em_rows, VSD_T, , true, kSampleToken)
                          : VSD_BY_RING(k_em_rows, VSD_T, , false, kSampleToken);
    cudaError_t e = prep(rows, smem);
    if (e) return e;
    if ((e = launch_after(rows, P.R, kThreads, smem, s, P)) || !grad) return e;
    return grad_rows(P, vec, grad, grad_bf16, s);
}

template <>
cudaError_t Launch<VSD_T>::verify_few(const Problem<VSD_T>& P, bool vec, cudaStream_t s) {
    const bool deep = deep_ring(vec, P.nch, P.R);
    const size_t smem = row_smem_bytes<sizeof(WeightsShared)>(P.nch, vec, deep);
    auto rows = VSD_BY_RING(k_em_rows, VSD_T, , false, kGivenToken);
    cudaError_t e = prep(rows, smem);
    if (e) return e;
    return launch_after(rows, P.R, kThreads, smem, s, P);
}

template <>
cudaError_t Launch<VSD_T>::grad_rows(const Problem<VSD_T>& P, bool vec, void* grad,
                                     bool grad_bf16, cudaStream_t s) {
    const bool kl = P.kl_topk != 0;
    // Gradient segments: a row each, or, where that leaves SMs short of blocks
    // (8 per SM keep about 64 KB in flight), several, of one batch of loads at
    // least.
    const long long nvec = (P.V + Traits<VSD_T>::kPerVec - 1) / Traits<VSD_T>::kPerVec;
    const long long batches = (nvec + kThreads * 8 - 1) / (kThreads * 8);
    long long nseg = ((long long)device_sm_count() * 8 + P.R - 1) / P.R;
    if (nseg > batches) nseg = batches;
    if (nseg < 1) nseg = 1;
#define VSD_EMG(V_, G_, K_)                                                                 \
    return launch_after(k_em_grad<VSD_T, V_, G_, K_>, (unsigned)(P.R * nseg), kThreads, 0, s, \
                        P, reinterpret_cast<G_*>(grad), (int)nseg)
#define VSD_EMG_KL(V_, G_)         \
    do {                           \
        if (kl) VSD_EMG(V_, G_, true); \
        VSD_EMG(V_, G_, false);    \
    } while (0)
    if (vec && grad_bf16) VSD_EMG_KL(true, __nv_bfloat16);
    if (vec) VSD_EMG_KL(true, float);
    if (grad_bf16) VSD_EMG_KL(false, __nv_bfloat16);
    VSD_EMG_KL(false, float);
#undef VSD_EMG_KL
#undef VSD_EMG
}

}  // namespace vsd
