// vsd_staged.cuh -- the E-step + M-step in two kernels (when: two_kernels() in
// vsd_api.cu):
//
//   k_em_rows  one block per row: the row pass (draws, statistics, the top-K
//              term of VSD (KL)).  The block completing a path's last row runs
//              the path (accepted length, residual draw, log-kappa sums), the
//              block completing a prefix's last path its M-step.  No block
//              waits for another.
//   k_em_grad  the gradient rows, as a programmatic dependent launch.
//
// Against the persistent kernel (k_fused) this gives up the overlap of one
// prefix's gradient with another's rows, and wins what claiming and handing
// over jobs costs: there a row's chain (claim, tail, path, M-step, publication,
// gradient claims) runs on one control warp per block while rows are short.
// Same results bit for bit.
//
// What bounds a single wave of rows (R up to 8 per SM) is the chain of one
// path: at 768 rows of V = 32000 the row streams 11 us, its tail takes 7, the
// path's residual draw 11, its epilogue 3, the M-step 9, the counters in
// between 2, the gradient 14 (65 us a call; 119 on the persistent kernel).
// Those steps run once per block and are short of instructions as much as of
// data, so loops in them are kept rolled.
#pragma once

#include "vsd_grid.cuh"
#include "vsd_launch.h"

namespace vsd {

// Dynamic shared memory: [ring][chunk table]; the M-step's scratch takes the
// place of the ring's chunk data, not of its barriers (vector rows), or follows
// the table.
inline size_t staged_smem_bytes(int nch, bool vec, bool deep) {
    return row_smem_bytes<sizeof(WeightsShared)>(nch, vec, deep) +
           (vec ? 0 : sizeof(WeightsShared));
}

// XMODE: kSampleToken the whole E-step + M-step; kGivenToken the verification
// of given tokens, which ends with the paths (few rows).
template <typename T, bool VEC, bool KL, int XMODE, int S>
__global__ void __launch_bounds__(kThreads, VEC ? kRowBlocks : 1) k_em_rows(Problem<T> P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ union {
        RowShared row;
        PathShared path;
    } sh;
    __shared__ int s_last;
    Ring<S>* rg;
    float4* tab;
    smem_views<VEC, sizeof(WeightsShared)>(dsm, rg, tab, P.timeout_ns, P.hold_copies != 0);
    grid_launch_next();
    const int r = blockIdx.x, D = P.D, K = P.K, nch = P.nch;
    const int64_t V = P.V;
    const T* x = P.draft + (int64_t)r * V;
    const T* y = P.target + (int64_t)r * V;
    const bool given = VEC && P.xtab_given;  // the LM head wrote the draft's half of the table
    if constexpr (VEC) {
        if (given)
            stream_target_tables<T>(rg, y, V, 0, nch, tab, P.ts.c, policy_evict_first(), P.status);
    }
    if (!given) {
        // (unaligned rows behind the LM head: that kernel still writes the logits)
        if (!VEC && P.xtab_given) grid_wait();
        stream_tables<T, VEC, true>(rg, x, y, V, 0, nch, tab, P.ts.c,
                                    P.gnseg ? policy_evict_last() : policy_evict_first(),
                                    policy_evict_first(), P.status);
    }
    // the kernel before this one (the clearing of the counters, or the LM
    // head) has ended; what was read so far is the call's input
    grid_wait();
    if (given) {
        const float4* rtab = P.gtab + (int64_t)r * P.nch_ws;
        for (int ch = threadIdx.x; ch < nch; ch += kThreads)
            reinterpret_cast<float2*>(tab + ch)[0] =
                __ldcg(reinterpret_cast<const float2*>(rtab + ch));
    }
    __syncthreads();
    row_tail<T, VEC, true, XMODE, true, KL>(P, r, tab, sh.row, rg);
    // the last of n blocks to arrive at a counter
    auto last_of = [&](int* cnt, int n) {
        __syncthreads();
        if (threadIdx.x == 0) s_last = atomic_add_acq_rel(cnt, 1) == n - 1;
        __syncthreads();
        return s_last != 0;
    };
    const int path = r / D;
    if (!last_of(P.path_cnt + path, D)) return;
    path_head<T>(P, path, sh.path);
    __syncthreads();
    const int A = sh.path.A, rA = path * D + A;
    int resid = -1;
    // (T = 0: the residual is the target's argmax, the row's p-draw)
    if (A < D && !sh.path.rec.flags && !P.greedy)
        resid = residual_draw<T, VEC>(P, rA, sh.path.rec, __ldg(P.u_correct + rA), rg, tab,
                                      &sh.path.resid);
    path_epilogue<T>(P, path, A, resid);
    if (XMODE == kGivenToken) return;
    const int prefix = path / K;
    if (!last_of(P.prefix_cnt + prefix, K)) return;
    WeightsShared* ws = VEC ? reinterpret_cast<WeightsShared*>(dsm)
                            : reinterpret_cast<WeightsShared*>(tab + nch);
    const EStepView E{P.es.tok, P.es.corr, P.es.lq_tok, P.es.lq_corr,
                      P.es.lk, P.es.lkc, P.es.lkr};
    weights_group<T, kThreads>(P, E, prefix, P.out.weights, P.out.loss, *ws, threadIdx.x);
    if (last_of(P.prefix_done, P.B) && threadIdx.x < 32)
        loss_mean(P.out.loss, P.B, threadIdx.x);
}

// The gradient of one segment of a row (block; nseg segments a row): the dense
// part g q(v) from eight 16-byte vectors in flight per thread (a row without
// one is not read), then the elements with sparse terms, one thread each, in
// the order of the persistent kernel's gradient jobs.
template <typename T, bool VEC, typename G, bool KL>
__global__ void __launch_bounds__(kThreads) k_em_grad(Problem<T> P, G* grad, int nseg) {
    __shared__ KlRec kl;
    constexpr int PV = Traits<T>::kPerVec, NP = PV / 2, U = 8;
    const int r = blockIdx.x / nseg, seg = blockIdx.x - r * nseg;
    const int64_t V = P.V;
    const T* x = P.draft + (int64_t)r * V;
    G* g = grad + (int64_t)r * V;
    const float c = P.ts.c;
    // segments are whole batches of the block's vectors
    const int nvec = (int)((V + PV - 1) / PV);
    const int per = ((nvec + nseg - 1) / nseg + kThreads - 1) / kThreads * kThreads;
    const int i0 = seg * per, i1 = min(nvec, i0 + per);
    grid_wait();
    const RowRec rec = ld_cg(P.rows + r);
    const Coef cf = ld_cg(P.coef + r);
    if (KL) {
        if (threadIdx.x < sizeof(KlRec) / 16)
            reinterpret_cast<int4*>(&kl)[threadIdx.x] =
                __ldcg(reinterpret_cast<const int4*>(P.klr + r) + threadIdx.x);
    }
    const float mx = rec.mx, gq = cf.g * rec.izx;  // g / Z
    const bool dense = !(cf.g == 0.f && isfinite(mx));
    // the logits with sparse terms, before the row is written (the gradient may
    // take the draft's place)
    const int j = (int)threadIdx.x - 2;
    int t = -1;
    if (j < 0)
        t = threadIdx.x ? cf.t1 : cf.t0;
    else if (KL && j < kMaxKlTop)
        t = ld_cg(&P.klr[r].tok[j]);
    const bool here = t >= i0 * PV && t < (int64_t)i1 * PV && t < V;
    const float xt = here && dense ? elem_value_cg(x, t) : 0.f;
    __syncthreads();
    if constexpr (VEC) {
        const uint64_t pol = policy_evict_first();
        const uint64_t mx2 = f2(mx, mx), c2 = f2(c, c), gq2 = f2(gq, gq);
        for (int ib = i0 + threadIdx.x; ib < i1; ib += kThreads * U) {
            uint4 buf[U];
            if (dense) {
#pragma unroll
                for (int k = 0; k < U; ++k)
                    if (ib + k * kThreads < i1)
                        buf[k] = ld_stream(x + (int64_t)(ib + k * kThreads) * PV, pol);
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const int i = ib + k * kThreads;
                if (i >= i1) break;
                float o[PV];
                if (dense) {
                    uint64_t pr[NP];
                    vec_pairs<T>(buf[k], pr);
#pragma unroll
                    for (int q = 0; q < NP; ++q)
                        f2split(f2mul(f2_mass(pr[q], mx2, c2), gq2), o[2 * q], o[2 * q + 1]);
                } else {
#pragma unroll
                    for (int e = 0; e < PV; ++e) o[e] = 0.f;
                }
                grad_store<T, G, PV>(g, (int64_t)i * PV, o, pol);
            }
        }
    } else {
        const int64_t e1 = min(V, (int64_t)i1 * PV);
        for (int64_t v = (int64_t)i0 * PV + threadIdx.x; v < e1; v += kThreads) {
            const float val =
                dense ? __fmul_rn(ex2(__fmul_rn(__fsub_rn(elem_value(x, v), mx), c)), gq) : 0.f;
            if constexpr (sizeof(G) == 2)
                g[v] = __float2bfloat16_rn(val);
            else
                g[v] = val;
        }
    }
    __syncthreads();
    // the elements with sparse terms: t0, t1, the top-K tokens
    const int nkl = KL ? min(max(kl.n, 0), kMaxKlTop) : 0;
    if ((int)threadIdx.x < 2 + nkl) {
        const bool mine = here && !(threadIdx.x >= 1 && t == cf.t0) &&
                          !(threadIdx.x >= 2 && t == cf.t1);
        if (mine) {
            // (rounded steps: no contraction into a fused multiply-add)
            float o = dense ? __fmul_rn(ex2(__fmul_rn(__fsub_rn(xt, mx), c)), gq) : 0.f;
            if (t == cf.t0) o = __fsub_rn(o, cf.c0);
            if (t == cf.t1) o = __fsub_rn(o, cf.c1);
            for (int k = 0; k < nkl; ++k)
                if (t == kl.tok[k]) o = __fadd_rn(o, kl.coef[k]);
            if constexpr (sizeof(G) == 2)
                g[t] = __float2bfloat16_rn(o);
            else
                g[t] = o;
        }
    }
}

}  // namespace vsd
