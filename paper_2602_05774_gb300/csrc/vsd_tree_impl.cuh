// vsd_tree_impl.cuh -- kernels and launchers of the draft trees for one logit
// dtype VSD_T.  Included once by vsd_tree_f32.cu and once by vsd_tree_bf16.cu.
#pragma once

#include "vsd_grid.cuh"
#include "vsd_launch.h"
#include "vsd_tree.cuh"

namespace vsd {

// ------------------------------------------------------------ fused tree kernel
// Tree verification in one launch of plain 128-thread blocks, R + tail
// blocks.  Each block first takes a ticket: a ticket below R is a node row
// (its tables and p-draw, then its children's acceptance; a leaf's row is
// skipped unless row statistics are requested); the block completing a
// tree's last row runs the per-node pass for that tree (its shared memory is
// the idle ring), queues the tree's residual rows and, when the bonus token
// needs the row of a leaf that was skipped, runs that row's pass itself as
// one more of the tree's items.  After its row a block takes queued residual
// rows (the rejected children's draws) while any are ready; the block
// completing a tree's last item writes its bonus token.  A block whose
// ticket is R or more was started after every row had
// been claimed, so every job it may wait for is held by a running block: it
// waits for residual rows (bounded, status bit on expiry) until every tree is
// done.
template <typename T>
__device__ int claim_residual(const Problem<T>& P, bool wait) {
    uint64_t idle_since = 0;
    for (;;) {
        const int it = *(volatile int*)P.resq_avail > 0
                           ? take_residual(P.resq_head, P.resq_avail, P.resq_flag, P.resq,
                                           P.status, P.timeout_ns)
                           : -1;
        if (it >= 0) return it;
        if (it == -2) return -1;
        if (!wait) return -1;
        if (*(volatile int*)P.prefix_done >= P.B) return -1;
        if (*(volatile int*)P.status & VSD_STATUS_TIMEOUT) return -1;
        const uint64_t now = global_timer_ns();
        if (idle_since == 0) {
            idle_since = now;
        } else if (now - idle_since > P.timeout_ns) {
            atomicOr(P.status, VSD_STATUS_TIMEOUT);
            return -1;
        }
        __nanosleep(1000);
    }
}

template <typename T, bool VEC>
__global__ void __launch_bounds__(kThreads) k_tree_fused(Problem<T> P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ RowShared sh;
    __shared__ int s_t, s_last, s_tok, s_cnt, s_leaf;
    Ring<kStages>* rg;
    float4* tab;
    smem_views<VEC>(dsm, rg, tab, P.timeout_ns);
    // The per-node pass runs between streams: on the vector path its shared
    // memory is the ring's data (no copy is in flight then), else it follows
    // the chunk table.
    static_assert(sizeof(TreeShared) <= sizeof(Ring<kStages>::data), "TreeShared fits the ring");
    TreeShared* tsh = VEC ? reinterpret_cast<TreeShared*>(rg->data)
                          : reinterpret_cast<TreeShared*>(tab + P.nch);
    const int N = P.N;
    grid_wait();
    if (threadIdx.x == 0) s_t = atomicAdd(P.ticket, 1);
    __syncthreads();
    const int t = s_t;
    if (t < P.R) {
        const int b = t / N, u = t - b * N;
        // A leaf's row is needed only for the bonus token (taken later if at
        // all) and for the row statistics output.
        int need = P.tout.row_stats != nullptr;
        for (int n = u + 1 + threadIdx.x; n < N && !need; n += kThreads)
            need = __ldg(P.parent + (int64_t)b * N + n) == u;
        if (__syncthreads_or(need)) {
            row_pass<T, VEC, true, kNoToken, false>(P, t, rg, tab, sh);
            __syncthreads();
            tree_children<T>(P, b, u);
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            __threadfence();
            s_last = atomicAdd(P.path_cnt + b, 1) == N - 1;
            if (s_last) __threadfence();
        }
        __syncthreads();
        if (s_last) {
            tree_nodes<T>(P, b, *tsh);
            __syncthreads();
            if (threadIdx.x == 0) {
                const int cnt = ld_cg(P.tcount + b);
                const int best = ld_cg(P.tout.deepest + b);
                const int child = best >= 0 ? ld_cg(P.tlist + b * N + N - 1) : 0;
                // a leaf's row not read yet that the bonus token needs
                const int leaf = (best >= 0 && child < 0 && !P.tout.row_stats) ? b * N + best : -1;
                s_cnt = cnt;
                s_leaf = leaf;
                if (cnt > 0) {  // queue the tree's residual rows (list positions)
                    // the leaf's row pass here counts as one more of the tree's items
                    if (leaf >= 0) atomicSub(P.res_seg_cnt + b, 1);
                    publish_residuals(P.resq_tail, P.resq_avail, P.resq_flag, P.resq, b * N,
                                      cnt, true);
                }
            }
            __syncthreads();
            const int cnt = s_cnt, leaf = s_leaf;
            if (leaf >= 0) {  // while other blocks take the residual rows
                row_pass<T, VEC, true, kNoToken, false>(P, leaf, rg, tab, sh);
                __syncthreads();
            }
            if (threadIdx.x == 0) {
                bool done = cnt == 0;
                if (!done && leaf >= 0) {
                    __threadfence();
                    done = atomicAdd(P.res_seg_cnt + b, 1) == cnt - 1;
                }
                if (done) {
                    __threadfence();
                    tree_bonus<T>(P, b);
                    __threadfence();
                    atomicAdd(P.prefix_done, 1);
                }
            }
            __syncthreads();
        }
    }
    const bool wait = t >= P.R;
    for (;;) {
        if (threadIdx.x == 0) s_t = claim_residual<T>(P, wait);
        __syncthreads();
        const int item = s_t;
        if (item < 0) break;
        const int b = item / N;
        tree_residual_row<T, VEC>(P, b, ld_cg(P.tlist + item), rg, tab, &s_tok);
        if (threadIdx.x == 0) {
            __threadfence();
            if (atomicAdd(P.res_seg_cnt + b, 1) == ld_cg(P.tcount + b) - 1) {
                __threadfence();
                tree_bonus<T>(P, b);
                __threadfence();
                atomicAdd(P.prefix_done, 1);
            }
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------ launchers
#ifndef VSD_TREE_TAIL_PER_SM
#define VSD_TREE_TAIL_PER_SM 1
#endif
template <>
cudaError_t Launch<VSD_T>::tree(const Problem<VSD_T>& P, bool vec, cudaStream_t s) {
    // one block per node row, then tail blocks for the last trees' residual rows
    const size_t smem = stream_smem_bytes<kStages>(P.nch, vec) + (vec ? 0 : sizeof(TreeShared));
    auto kern = vec ? k_tree_fused<VSD_T, true> : k_tree_fused<VSD_T, false>;
    cudaError_t e = prep(kern, smem);
    if (e) return e;
    long long tail = (long long)device_sm_count() * VSD_TREE_TAIL_PER_SM;
    const long long most = (long long)P.B * (P.N - 1);  // residual rows at most
    if (tail > most) tail = most;
    if (tail < 1) tail = 1;
    return launch_after(kern, (unsigned)(P.R + tail), kThreads, smem, s, P);
}

template <>
cudaError_t Launch<VSD_T>::tree_seq(const Problem<VSD_T>& P, bool vec, cudaStream_t s) {
    const size_t smem = stream_smem_bytes<kRowStages>(P.nch, vec) + seq_smem_bytes(P.N);
    auto rows = vec ? k_tree_seq_rows<VSD_T, true> : k_tree_seq_rows<VSD_T, false>;
    cudaError_t e = prep(rows, smem);
    if (e) return e;
    if ((e = launch_after(rows, P.R, kThreads, smem, s, P))) return e;
    const size_t sm2 = stream_smem_bytes<kRowStages>(P.nch, vec) + sizeof(TreeSeqShared);
    auto seq = vec ? k_tree_seq<VSD_T, true> : k_tree_seq<VSD_T, false>;
    if ((e = prep(seq, sm2))) return e;
    return launch_after(seq, P.B, kThreads, sm2, s, P);
}

template <>
cudaError_t Launch<VSD_T>::tree_em(const Problem<VSD_T>& P, bool vec,
                                   const vsd_tree_em_outputs& o, void* grad, bool grad_bf16,
                                   cudaStream_t s) {
    const size_t smem = stream_smem_bytes<kRowStages>(P.nch, vec);
    auto rows = vec ? k_tree_rows<VSD_T, true> : k_tree_rows<VSD_T, false>;
    cudaError_t e = prep(rows, smem);
    if (e) return e;
    if ((e = launch_after(rows, P.R, kThreads, smem, s, P))) return e;
    auto draws = vec ? k_tree_draws<VSD_T, true> : k_tree_draws<VSD_T, false>;
    if ((e = prep(draws, smem))) return e;
    if ((e = launch_after(draws, P.R, kThreads, smem, s, P))) return e;
    if ((e = prep(k_tree_em<VSD_T>, sizeof(TreeEmShared)))) return e;
    if ((e = launch_after(k_tree_em<VSD_T>, P.B, kThreads, sizeof(TreeEmShared), s, P, o)))
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
