// vsd_tree_impl.cuh -- kernels and launchers of the draft trees for one logit
// dtype VSD_T.  Included once by vsd_tree_f32.cu and once by vsd_tree_bf16.cu.
#pragma once

#include "vsd_grid.cuh"
#include "vsd_launch.h"
#include "vsd_tree.cuh"

namespace vsd {

// ------------------------------------------------------------ launchers
template <>
cudaError_t Launch<VSD_T>::tree(const Problem<VSD_T>& P, bool vec, cudaStream_t s) {
    const bool deep = deep_ring(vec, P.nch, P.R);
    const size_t smem = row_smem_bytes(P.nch, vec, deep);
    auto rows = VSD_BY_RING(k_tree_verify_rows, VSD_T);
    cudaError_t e = prep(rows, smem);
    if (e) return e;
    if ((e = launch_after(rows, P.R, kThreads, smem, s, P))) return e;
    const size_t sm2 = smem + tree_verify_smem_bytes(P.N);
    auto nodes = P.tout.row_stats ? VSD_BY_RING(k_tree_verify, VSD_T, , true)
                                  : VSD_BY_RING(k_tree_verify, VSD_T, , false);
    if ((e = prep(nodes, sm2))) return e;
    return launch_after(nodes, P.R, kThreads, sm2, s, P);
}

template <>
cudaError_t Launch<VSD_T>::tree_seq(const Problem<VSD_T>& P_, bool vec, cudaStream_t s) {
    Problem<VSD_T> P = P_;
    P.read_leaves = P.R <= device_sm_count();
    const bool deep = deep_ring(vec, P.nch, P.R);
    const size_t smem = row_smem_bytes(P.nch, vec, deep) + seq_smem_bytes(P.N);
    auto rows = VSD_BY_RING(k_tree_seq_rows, VSD_T);
    cudaError_t e = prep(rows, smem);
    if (e) return e;
    if ((e = launch_after(rows, P.R, kThreads, smem, s, P))) return e;
    const size_t sm2 = row_smem_bytes(P.nch, vec, deep) + sizeof(TreeSeqShared);
    auto seq = VSD_BY_RING(k_tree_seq, VSD_T);
    if ((e = prep(seq, sm2))) return e;
    return launch_after(seq, P.B, kThreads, sm2, s, P);
}

template <>
cudaError_t Launch<VSD_T>::tree_em(const Problem<VSD_T>& P, bool vec,
                                   const vsd_tree_em_outputs& o, void* grad, bool grad_bf16,
                                   cudaStream_t s) {
    const bool deep = deep_ring(vec, P.nch, P.R);
    const size_t smem = row_smem_bytes(P.nch, vec, deep);
    auto rows = VSD_BY_RING(k_tree_rows, VSD_T);
    cudaError_t e = prep(rows, smem);
    if (e) return e;
    if ((e = launch_after(rows, P.R, kThreads, smem, s, P))) return e;
    auto draws = VSD_BY_RING(k_tree_draws, VSD_T);
    if ((e = prep(draws, smem))) return e;
    if ((e = launch_after(draws, P.R, kThreads, smem, s, P))) return e;
    if ((e = prep(k_tree_em<VSD_T>, sizeof(TreeEmShared)))) return e;
    if ((e = launch_after(k_tree_em<VSD_T>, P.B, kEmThreads, sizeof(TreeEmShared), s, P, o)))
        return e;
    const size_t gsm = tree_grad_smem_bytes(P.N);
#define VSD_TGRAD(V_, G_)                                                           \
    do {                                                                            \
        if ((e = prep(k_tree_grad<VSD_T, V_, G_>, gsm))) return e;                  \
        return launch_after(k_tree_grad<VSD_T, V_, G_>, P.R, kThreads, gsm, s, P,   \
                            reinterpret_cast<G_*>(grad));                           \
    } while (0)
    if (vec && grad_bf16) VSD_TGRAD(true, __nv_bfloat16);
    else if (vec) VSD_TGRAD(true, float);
    else if (grad_bf16) VSD_TGRAD(false, __nv_bfloat16);
    else VSD_TGRAD(false, float);
#undef VSD_TGRAD
}

}  // namespace vsd
