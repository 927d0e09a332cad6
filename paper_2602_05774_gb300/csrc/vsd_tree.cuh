// vsd_tree.cuh -- draft trees beyond independent branch verification (App. E
// trees): the E-step + M-step with every node a latent proposal, and tree
// verification with the sequential sibling rule (lossless multi-draft).
//
//   k_tree_rows  one block per node row u: the row pass (tables, statistics,
//                the target's argmax), then for every child x of u its token's
//                test at u's row (Eq. 1, each branch alone).
//   k_tree_draws one block per row with children: the draws their corrected
//                paths take there, from the residual norm(max(0, p - q)) at
//                the first rejection, from p below it.
//   k_tree_em    one block per tree: the accepted paths, the corrected path
//                z' of every node, the log-kappa sums along the root paths
//                (Eq. 2), o~ and o' (Algorithm 2), beta and zeta over the nodes
//                of one depth (Eqs. beta, zeta), the loss (Eq. advance) and
//                each node's gradient terms (sums over its subtree).
//   k_tree_grad  one block per row: grad = g q(v) minus the sparse terms of
//                the row's children (their tokens and corrected tokens).
//   k_tree_seq_rows / k_tree_seq   the sequential sibling rule: one block per
//                row decides which of the row's children is accepted, one block
//                per tree follows the decisions along the accepted path.
#pragma once

#include "vsd_passes.cuh"

namespace vsd {

// What k_tree_rows leaves for a node x (at index b*N + x).
struct __align__(16) TreeNodeRec {
    float la;      // log alpha of x's token at its parent's row (the branch alone)
    float lq;      // log q of that token
    int acc;       // u_accept <= alpha
    int zp;        // draw from p at the parent's row with x's u_correct (-1: none)
    float lq_zp, la_zp;
    int zr;        // residual draw at the parent's row with x's u_correct (-1: none)
    float lq_zr, la_zr;
    int pad[3];
};
static_assert(sizeof(TreeNodeRec) == 48, "TreeNodeRec layout");

// A node's gradient terms at its parent's row, scaled by 1 / (B N_b T):
// -ct at its token t, -cz at its corrected token z (z = -1: none).
struct __align__(16) TreeCoef {
    int t;
    float ct;
    int z;
    float cz;
};
static_assert(sizeof(TreeCoef) == 16, "TreeCoef layout");

// ------------------------------------------------------------ verification
// Every branch alone (VSD_TREE_INDEPENDENT), two kernels:
//   k_tree_verify_rows  one block per node row with children (any row for the
//                       statistics output): the row's statistics, then each
//                       child's test;
//   k_tree_verify       one block per row, of which most leave at once: at a
//                       row on an accepted path the rejected children's draws
//                       (one more read of the row), at the deepest accepted
//                       node the bonus token (a leaf's row is read here, or
//                       its chunk table if the first kernel read it), at the root
//                       the outputs of the tree's nodes.
// No block waits for another.  The row reads bound the first kernel, a few
// dependent steps of one row the second.
template <typename T, bool VEC, int S>
__global__ void __launch_bounds__(kThreads, VEC ? kRowBlocks : 1)
    k_tree_verify_rows(Problem<T> P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ RowShared sh;
    Ring<S>* rg;
    float4* tab;
    smem_views<VEC>(dsm, rg, tab, P.timeout_ns, P.hold_copies != 0);
    grid_launch_next();
    const int r = blockIdx.x, N = P.N, b = r / N, u = r - b * N;
    int kids = 0;
    for (int n = u + 1 + threadIdx.x; n < N && !kids; n += kThreads)
        kids = __ldg(P.parent + (int64_t)b * N + n) == u;
    kids = __syncthreads_or(kids);
    if (!kids && !P.tout.row_stats) {
        grid_wait();
        return;
    }
    row_pass<T, VEC, true, kStats, false>(P, r, rg, tab, sh);
    __syncthreads();
    if (!kids) {  // the table for a bonus token drawn here
        for (int ch = threadIdx.x; ch < P.nch; ch += kThreads)
            P.gtab[(int64_t)r * P.nch_ws + ch] = tab[ch];
    }
    tree_children<T>(P, b, u);
}

// Per node of the tree (dynamic shared memory, after the chunk table).
struct TreeVerifyNodes {
    double* lk;  // [N] log kappa
    int* par;
    int* depth;  // -1: not on an accepted path (every node's at the root's block)
    float* la;
    unsigned char* acc;
};
inline size_t tree_verify_smem_bytes(int N) { return (size_t)N * 21 + 16; }

// STATS: with row_stats (the first kernel has read every row).
template <typename T, bool VEC, bool STATS, int S>
__global__ void __launch_bounds__(kThreads) k_tree_verify(Problem<T> P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ RowShared sh;
    __shared__ int s_path, s_best, s_maxd, s_any, s_more, s_first;
    Ring<S>* rg;
    float4* tab;
    smem_views<VEC>(dsm, rg, tab, P.timeout_ns, P.hold_copies != 0);
    const int r = blockIdx.x, N = P.N, b = r / N, u = r - b * N, n0 = b * N;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const vsd_tree_outputs& o = P.tout;
    TreeVerifyNodes t;
    t.lk = reinterpret_cast<double*>(tab + P.nch);
    t.par = reinterpret_cast<int*>(t.lk + N);
    t.depth = t.par + N;
    t.la = reinterpret_cast<float*>(t.depth + N);
    t.acc = reinterpret_cast<unsigned char*>(t.la + N);
    int bad = 0;
    for (int n = tid; n < N; n += kThreads) {
        const int pn = __ldg(P.parent + n0 + n);
        t.par[n] = pn;
        bad |= n == 0 ? pn != -1 : (pn < 0 || pn >= n);
    }
    grid_wait();
    if (__syncthreads_or(bad)) {
        if (u) return;
        for (int n = tid; n < N; n += kThreads) {
            o.alpha[n0 + n] = 0.f;
            o.accept[n0 + n] = 0;
            o.path_accept[n0 + n] = 0;
            o.logkappa[n0 + n] = -INFINITY;
            o.corr_tokens[n0 + n] = -1;
        }
        if (tid == 0) {
            atomicOr(P.status, VSD_STATUS_BAD_TREE);
            o.deepest[b] = -1;
            o.accept_len[b] = -1;
            o.bonus[b] = -1;
        }
        return;
    }
    int* up = t.depth;  // (for now) an accepted node's parent, -1 for a rejected one
    for (int n = tid; n < N; n += kThreads) {
        const int acc = n ? ld_cg(o.accept + n0 + n) : 1;
        t.acc[n] = acc;
        up[n] = acc ? t.par[n] : -1;
        if (u == 0) t.la[n] = n ? ld_cg(P.tla + n0 + n) : 0.f;
    }
    __syncthreads();
    if (tid == 0) {
        int x = u;
        while (x > 0) x = up[x];
        s_path = x == 0;
        s_best = -1;
        s_maxd = s_any = s_more = 0;
        s_first = N;
    }
    __syncthreads();
    if (!s_path) return;
    auto child = [&](int n) {
        if (n <= u || t.par[n] != u) return;
        atomicMin(&s_first, n);
        if (t.acc[n]) s_more = 1;
        else s_any = 1;
    };
    // n's depth (-1 - it below a rejection) and, over the nodes, the deepest
    // accepted one (lowest index on ties), for the nodes' outputs and for the bonus
    // token.  Each node walks to the root, so only the root's block and those of
    // nodes without an accepted child take it (64 chains of 1024 accepted nodes:
    // 14.7 ms a call with it in every block on an accepted path, 2.8 now).
    auto walk = [&](int n) {
        int d = 0, ok = 1;
        for (int x = n; x > 0; x = t.par[x]) {
            ok &= t.acc[x];
            ++d;
        }
        t.depth[n] = ok ? d : -1 - d;
        if (ok) atomicMax(&s_best, (d << 11) | (2047 - n));
        atomicMax(&s_maxd, d);
    };
    for (int n = tid; n < N; n += kThreads) {
        child(n);
        if (u == 0) walk(n);
    }
    __syncthreads();
    if (u && !s_more) {
        for (int n = tid; n < N; n += kThreads) walk(n);
        __syncthreads();
    }
    const int best = s_best < 0 ? -1 : 2047 - (s_best & 2047);
    if (u == 0) {  // the nodes' outputs; log kappa along each branch (Eq. 2)
        auto depth_of = [&](int n) { return t.depth[n] >= 0 ? t.depth[n] : -1 - t.depth[n]; };
        for (int l = 0; l <= s_maxd; ++l) {
            for (int n = tid; n < N; n += kThreads)
                if (depth_of(n) == l) t.lk[n] = n ? t.lk[t.par[n]] + (double)t.la[n] : 0.0;
            __syncthreads();
        }
        for (int n = tid; n < N; n += kThreads) {
            const bool pa = t.depth[n] >= 0;
            o.path_accept[n0 + n] = pa;
            o.logkappa[n0 + n] = (float)t.lk[n];
            // (a rejected child of an accepted node: its parent's block draws)
            if (pa || t.depth[t.par[n]] < 0) o.corr_tokens[n0 + n] = -1;
        }
        if (tid == 0) {
            o.alpha[n0] = 1.f;
            o.accept[n0] = 1;
            o.deepest[b] = best;
            o.accept_len[b] = t.depth[best];
        }
    }
    const int64_t V = P.V;
    if (s_any) {  // the rejected children's draws from norm(max(0, p - q))
        const RowRec rec = ld_cg(P.rows + r);
        const T* x = P.draft + (int64_t)r * V;
        const T* y = P.target + (int64_t)r * V;
        const float c = P.ts.c;
        const uint64_t pol = policy_evict_normal();
        const MassRes mr{rec.mx, rec.my, rec.izx, rec.izy, c};
        TableSum R{0, 0, 0.0}, Sp{0, 0, 0.0};
        float M = 0.f;
        if (!rec.flags) {
            stream_residual<T, VEC>(rg, x, y, V, 0, P.nch, tab, mr, P.status);
            __syncthreads();
            R = table_sum(tab, P.nch, 0, 0.f, c, lane);
            if (!(R.Z > 0.0)) {  // no residual mass: draws from p with the same uniforms
                __syncthreads();
                stream_tables<T, VEC, false>(rg, y, nullptr, V, 0, P.nch, tab, c, pol, pol,
                                             P.status);
                __syncthreads();
                M = table_max(tab, P.nch, 0, lane);
                Sp = table_sum(tab, P.nch, 0, frame_of(M), c, lane);
            }
        }
        int k = 0;
        for (int n = u + 1; n < N; ++n) {
            if (t.par[n] != u || t.acc[n] || k++ % kWarps != warp) continue;
            const float uc = __ldg(P.u_correct + n0 + n);
            int tok = -1;
            if (R.Z > 0.0) {
                const Located loc = table_locate(tab, P.nch, 0, 0.f, c, R, uc, lane);
                if (loc.ch >= 0)
                    tok = warp_rescan<T, VEC, true, true>(x, y, V, loc.ch, loc.tc, mr, lane, pol,
                                                          warp_chunks(rg));
            } else if (row_ok(M, Sp.Z)) {
                tok = warp_sample<T, VEC>(y, nullptr, V, tab, P.nch, 0, M, Sp, uc, c, lane, pol,
                                          warp_chunks(rg));
            }
            if (lane == 0) o.corr_tokens[n0 + n] = tok < V ? tok : -1;
        }
        __syncthreads();
    }
    if (u == best) {  // the token after the accepted path
        const bool leaf = s_first == N;
        if (STATS && leaf) {  // its statistics are there, and its chunk table
            for (int ch = tid; ch < P.nch; ch += kThreads)
                tab[ch] = ld_cg(P.gtab + (int64_t)r * P.nch_ws + ch);
            __syncthreads();
            if (warp == 0) {
                const float M = table_max(tab, P.nch, 1, lane);
                const TableSum Sp = table_sum(tab, P.nch, 1, frame_of(M), P.ts.c, lane);
                int tok = -1;
                if (!ld_cg(P.rows + r).flags)
                    tok = warp_sample<T, VEC>(P.draft + (int64_t)r * V, P.target + (int64_t)r * V, V,
                                              tab, P.nch, 1, M, Sp, __ldg(P.u_correct + r), P.ts.c,
                                              lane, policy_evict_normal(), warp_chunks(rg));
                if (lane == 0) o.bonus[b] = tok < V ? tok : -1;
            }
            return;
        }
        if (leaf) {
            row_pass<T, VEC, true, kNoToken, false>(P, r, rg, tab, sh);
            __syncthreads();
        }
        if (tid == 0)
            o.bonus[b] = leaf ? ld_cg(P.rows + r).ps : ld_cg(o.corr_tokens + n0 + s_first);
    }
}

// ------------------------------------------------------------ k_tree_rows
// One block per node row: the row pass, then each child's token tested at the
// row (one thread per child: Eq. 1, each branch alone), and the row's chunk
// table kept in global memory for the draws.
template <typename T, bool VEC, int S>
__global__ void __launch_bounds__(kThreads, VEC ? kRowBlocks : 1) k_tree_rows(Problem<T> P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ RowShared sh;
    Ring<S>* rg;
    float4* tab;
    smem_views<VEC>(dsm, rg, tab, P.timeout_ns, P.hold_copies != 0);
    grid_launch_next();
    const int r = blockIdx.x, N = P.N, b = r / N, u = r - b * N, n0 = b * N;
    const int64_t V = P.V;
    row_pass<T, VEC, true, kStats, true>(P, r, rg, tab, sh);
    __syncthreads();
    const RowRec rec = ld_cg(P.rows + r);
    int kids = 0;
    for (int n = u + 1 + threadIdx.x; n < N; n += kThreads) {
        if (__ldg(P.parent + n0 + n) != u) continue;
        kids = 1;
        TreeNodeRec nr;
        nr.la = nr.lq = -INFINITY;
        nr.zp = nr.zr = -1;
        nr.lq_zp = nr.la_zp = nr.lq_zr = nr.la_zr = -INFINITY;
        nr.pad[0] = nr.pad[1] = nr.pad[2] = 0;
        const int tok = __ldg(P.given_tokens + n0 + n);
        if (tok < 0 || tok >= V)
            atomicOr(P.status, VSD_STATUS_BAD_TOKEN);
        else if (!rec.flags)
            token_logs(P.draft + (int64_t)r * V, P.target + (int64_t)r * V, tok, rec, P.ts.invTd,
                       &nr.lq, &nr.la);
        nr.acc = nr.la > -INFINITY && __ldg(P.u_accept + n0 + n) <= expf(nr.la);
        P.tnode[n0 + n] = nr;
    }
    if (__syncthreads_or(kids))
        for (int ch = threadIdx.x; ch < P.nch; ch += kThreads)
            P.gtab[(int64_t)r * P.nch_ws + ch] = tab[ch];
}

// ------------------------------------------------------------ k_tree_draws
// One block per row with children: the corrected tokens its children may
// need, and no others.  On an accepted path a rejected child draws from the
// row's residual max(0, p - q) (one more read of the row; from p if that has
// no mass); below a rejection every child draws from p, for which the row's
// chunk table and one chunk suffice.  Whether u is on an accepted path follows
// from the acceptance bits of its ancestors, which are all known here; only
// these few rows are read twice (64 trees of 60 nodes: about 300 of 3840).
template <typename T, bool VEC, int S>
__global__ void __launch_bounds__(kThreads) k_tree_draws(Problem<T> P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ int s_par[1024], s_path;
    __shared__ unsigned char s_acc[1024];
    Ring<S>* rg;
    float4* tab;
    smem_views<VEC>(dsm, rg, tab, P.timeout_ns, P.hold_copies != 0);
    grid_launch_next();
    const int r = blockIdx.x, N = P.N, b = r / N, u = r - b * N, n0 = b * N;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int kids = 0;
    for (int n = threadIdx.x; n < N; n += kThreads) {
        const int pn = __ldg(P.parent + n0 + n);
        s_par[n] = pn;
        kids |= n > u && pn == u;
    }
    grid_wait();
    if (!__syncthreads_or(kids)) return;
    for (int n = threadIdx.x; n < N; n += kThreads)
        s_acc[n] = n ? ld_cg(&P.tnode[n0 + n].acc) != 0 : 1;
    __syncthreads();
    if (threadIdx.x == 0) {
        int path = 1, x = u;
        while (x > 0 && path > 0) {
            const int pn = s_par[x];
            path = pn < 0 || pn >= x ? -1 : s_acc[x];  // -1: a bad tree
            x = pn;
        }
        s_path = path;
    }
    __syncthreads();
    const int path = s_path;
    const RowRec rec = ld_cg(P.rows + r);
    if (path < 0 || rec.flags) return;
    const int64_t V = P.V;
    const T* x = P.draft + (int64_t)r * V;
    const T* y = P.target + (int64_t)r * V;
    const float c = P.ts.c;
    const uint64_t pol = policy_evict_normal();
    const double invT = P.ts.invTd;
    // f(n) for the children that need a draw, shared out among the warps
    auto each_child = [&](auto&& f) {
        int k = 0;
        for (int n = u + 1; n < N; ++n)
            if (s_par[n] == u && !(path && s_acc[n]) && k++ % kWarps == warp)
                f(n0 + n);
    };
    if (path) {
        int rej = 0;
        for (int n = u + 1 + threadIdx.x; n < N; n += kThreads)
            rej |= s_par[n] == u && !s_acc[n];
        if (!__syncthreads_or(rej)) return;
        const MassRes mr{rec.mx, rec.my, rec.izx, rec.izy, c};
        stream_residual<T, VEC>(rg, x, y, V, 0, P.nch, tab, mr, P.status);
        __syncthreads();
        const TableSum Rt = table_sum(tab, P.nch, 0, 0.f, c, lane);
        if (Rt.Z > 0.0) {
            each_child([&](int n) {
                const Located loc =
                    table_locate(tab, P.nch, 0, 0.f, c, Rt, __ldg(P.u_correct + n), lane);
                if (loc.ch < 0) return;
                const int z = warp_rescan<T, VEC, true, true>(x, y, V, loc.ch, loc.tc, mr, lane,
                                                              pol, warp_chunks(rg));
                if (z < 0 || z >= V) return;
                float lq, la;
                token_logs(x, y, z, rec, invT, &lq, &la);
                if (lane == 0) {
                    P.tnode[n].zr = z;
                    P.tnode[n].lq_zr = lq;
                    P.tnode[n].la_zr = la;
                }
            });
            return;
        }
        __syncthreads();  // no residual mass: draws from p with the same uniforms
    }
    for (int ch = threadIdx.x; ch < P.nch; ch += kThreads)
        tab[ch] = ld_cg(P.gtab + (int64_t)r * P.nch_ws + ch);
    __syncthreads();
    const float My = table_max(tab, P.nch, 1, lane);
    const TableSum Sy = table_sum(tab, P.nch, 1, frame_of(My), c, lane);
    each_child([&](int n) {
        const int z = warp_sample<T, VEC>(x, y, V, tab, P.nch, 1, My, Sy, __ldg(P.u_correct + n), c,
                                          lane, pol, warp_chunks(rg));
        if (z < 0 || z >= V) return;
        float lq, la;
        token_logs(x, y, z, rec, invT, &lq, &la);
        if (lane == 0) {
            TreeNodeRec* nr = P.tnode + n;
            (path ? nr->zr : nr->zp) = z;
            (path ? nr->lq_zr : nr->lq_zp) = lq;
            (path ? nr->la_zr : nr->la_zp) = la;
        }
    });
}

// ------------------------------------------------------------ shared helpers
struct TreeShared2 {
    int par[1024];
    int depth[1024];
    short anc[1024];
    unsigned char pacc[1024];
    int maxd;
};

// Parents into shared memory and the tree's checks (parent[0] = -1, every
// other parent precedes its node); depths.  Returns false for a bad tree.
template <int NT, typename T>
__device__ bool tree_load(const Problem<T>& P, int b, TreeShared2& sh) {
    const int N = P.N;
    const int32_t* par = P.parent + (int64_t)b * N;
    int badl = 0;
    for (int n = threadIdx.x; n < N; n += NT) {
        const int pn = __ldg(par + n);
        sh.par[n] = pn;
        badl |= n == 0 ? pn != -1 : (pn < 0 || pn >= n);
    }
    const int bad = __syncthreads_or(badl);
    if (bad) return false;
    // depths by pointer doubling: depth[n] steps from n to anc[n]
    for (int n = threadIdx.x; n < N; n += NT) {
        sh.depth[n] = n ? 1 : 0;
        sh.anc[n] = (short)(n ? sh.par[n] : 0);
    }
    if (threadIdx.x == 0) sh.maxd = 0;
    for (;;) {
        __syncthreads();
        short a[1024 / NT];
        int d[1024 / NT];
        int more = 0;
#pragma unroll
        for (int k = 0; k < 1024 / NT; ++k) {
            const int n = threadIdx.x + k * NT;
            if (n >= N) break;
            a[k] = sh.anc[sh.anc[n]];
            d[k] = sh.depth[n] + sh.depth[sh.anc[n]];
            more |= a[k] != 0;
        }
        more = __syncthreads_or(more);
#pragma unroll
        for (int k = 0; k < 1024 / NT; ++k) {
            const int n = threadIdx.x + k * NT;
            if (n >= N) break;
            sh.anc[n] = a[k];
            sh.depth[n] = d[k];
        }
        if (!more) break;
    }
    __syncthreads();
    int md = 0;
    for (int n = threadIdx.x; n < N; n += NT) md = max(md, sh.depth[n]);
    atomicMax(&sh.maxd, md);
    __syncthreads();
    return true;
}

// ------------------------------------------------------------ k_tree_em
// The M-step of one tree, in double precision, by one block: the sums along
// the root paths go level by level (a node adds its term to its parent's sum),
// the subtree sums back up level by level (a node adds its children's sums in
// descending node order), and what belongs to one node or one depth is taken
// in parallel.  The order of every sum is fixed, so the result does not depend
// on scheduling.  (On one thread per tree the fp64 latency of this pass was
// 578 us of a call's 873 at 64 trees of 60 nodes; the whole call now takes 210,
// this pass about 25.)
// (256 threads are no faster at 60 nodes, 512 slower: 40.7, 40.0, 45.0 us)
constexpr int kEmThreads = 128, kEmWarps = kEmThreads / 32;
struct TreeEmShared {
    TreeShared2 t;
    double lk[1024], lkc[1024], lkr[1024], lqt[1024], lqz[1024];
    union {
        struct {
            float la[1024], laz[1024], lar[1024], lq[1024];  // the nodes' own terms
        } e;
        struct {
            double st[1024], sz[1024];  // CAR logits, then subtree sums of the gradient terms
        } m;
    };
    float w[1024][4];            // o~, o', beta, zeta
    float lqzn[1024];            // log q of z'_x at its parent's row
    int z[1024];                 // corrected token z'_x
    unsigned char acc[1024];
    short first[1024], last[1024];  // a node's first and last child (0: none)
    short prev[1024], next[1024];   // a node's siblings before and after it (0: none)
    // per depth: proposals with o' != 0 and o~ = 1, with o' != 0; the largest
    // CAR logit (as an ordered integer); the sum of the CAR weights
    int n1[1024], n0[1024];
    unsigned long long cmax[1024];
    double zs[1024];
    double red[kEmWarps][2];
};

// Doubles as integers of the same order (0 is below every double).
__device__ __forceinline__ unsigned long long ordered_bits(double v) {
    const long long b = __double_as_longlong(v);
    return b < 0 ? ~(unsigned long long)b : (unsigned long long)b | 0x8000000000000000ull;
}
__device__ __forceinline__ double ordered_value(unsigned long long k) {
    return __longlong_as_double(
        (long long)(k >> 63 ? k & 0x7FFFFFFFFFFFFFFFull : ~k));
}

// Sum over the block in a fixed order; every thread returns it.
__device__ __forceinline__ double2 block_sum(double2 v, double (*red)[2]) {
    v.x = warp_sum(v.x);
    v.y = warp_sum(v.y);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5][0] = v.x;
        red[threadIdx.x >> 5][1] = v.y;
    }
    __syncthreads();
    double2 s = make_double2(0.0, 0.0);
    for (int w = 0; w < kEmWarps; ++w) {
        s.x += red[w][0];
        s.y += red[w][1];
    }
    return s;
}

template <typename T>
__device__ void tree_em_nodes(const Problem<T>& P, const vsd_tree_em_outputs& o, int b,
                              TreeEmShared& sh) {
    const int N = P.N, n0 = b * N, tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int* par = sh.t.par;
    const int* depth = sh.t.depth;
    const int maxd = sh.t.maxd;
    for (int n = tid; n < N; n += kEmThreads) {
        sh.acc[n] = n ? P.tnode[n0 + n].acc != 0 : 1;
        sh.first[n] = sh.last[n] = 0;
        sh.n0[n] = sh.n1[n] = 0;
        sh.cmax[n] = 0;
    }
    // accepted paths
    for (int l = 0; l <= maxd; ++l) {
        __syncthreads();
        for (int n = tid; n < N; n += kEmThreads)
            if (depth[n] == l) sh.t.pacc[n] = n ? sh.acc[n] && sh.t.pacc[par[n]] : 1;
    }
    __syncthreads();
    // the E-step per node (R15): z' and the node's terms of the sums
    for (int n = tid; n < N; n += kEmThreads) {
        if (n == 0) {
            sh.lk[0] = sh.lkc[0] = sh.lkr[0] = sh.lqt[0] = sh.lqz[0] = 0.0;
            sh.z[0] = -1;
            sh.lqzn[0] = 0.f;
            continue;
        }
        const int a = par[n];
        const TreeNodeRec nr = ld_cg_rec(P.tnode + n0 + n);
        const RowRec ra = ld_cg(P.rows + n0 + a);
        int zc;
        float lqz, laz;
        if (sh.t.pacc[n]) {
            zc = __ldg(P.given_tokens + n0 + n); lqz = nr.lq; laz = nr.la;
        } else if (sh.t.pacc[a]) {  // the first rejection on the path: the residual
            zc = nr.zr; lqz = nr.lq_zr; laz = nr.la_zr;
        } else {                    // below a rejection: the draw from p
            zc = nr.zp; lqz = nr.lq_zp; laz = nr.la_zp;
        }
        if (zc < 0) { lqz = -INFINITY; laz = -INFINITY; }
        sh.z[n] = zc;
        sh.lqzn[n] = lqz;
        sh.e.la[n] = nr.la;
        sh.e.laz[n] = laz;
        sh.e.lar[n] = (ra.flags || ra.ref < 0) ? -INFINITY : ra.la_ref;
        sh.e.lq[n] = nr.lq;
        if (o.logq_tok) o.logq_tok[n0 + n] = nr.lq;
    }
    for (int l = 1; l <= maxd; ++l) {
        __syncthreads();
        for (int n = tid; n < N; n += kEmThreads) {
            if (depth[n] != l) continue;
            const int a = par[n];
            sh.lk[n] = sh.lk[a] + (double)sh.e.la[n];
            sh.lkc[n] = sh.lkc[a] + (double)sh.e.laz[n];
            sh.lkr[n] = sh.lkr[a] + (double)sh.e.lar[n];
            sh.lqt[n] = sh.lqt[a] + (double)sh.e.lq[n];
            sh.lqz[n] = sh.lqz[a] + (double)sh.lqzn[n];
        }
    }
    __syncthreads();
    // o~, o' (Algorithm 2 with w(depth): w(l) = w_base^l, trees may be deeper
    // than the host's table of w), N_b, the CAR logits
    double2 Nb = make_double2(0.0, 0.0);
    for (int n = 1 + tid; n < N; n += kEmThreads) {
        const double wl = depth[n] <= 64 ? P.wl[depth[n] - 1] : pow(P.w_base, (double)depth[n]);
        const bool ot = sh.lk[n] >= sh.lkr[n];
        const bool op = ot || sh.lkc[n] >= sh.lkr[n];
        sh.w[n][0] = ot ? 1.f : 0.f;
        sh.w[n][1] = op ? (float)wl : 0.f;
        const double cq = (P.zeta_mode == 0 ? exp(sh.lqt[n]) : sh.lqt[n]) * P.inv_tau;
        sh.m.st[n] = cq;
        const int l = depth[n] - 1;
        atomicMax(&sh.cmax[l], ordered_bits(cq));
        if (op) {
            Nb.x += wl;
            atomicAdd(&sh.n0[l], 1);
            if (ot) atomicAdd(&sh.n1[l], 1);
        }
    }
    Nb = block_sum(Nb, sh.red);
    // beta (leave-one-out) and zeta (softmax of q(z~)/tau, or log q in
    // zeta_mode 1) over the nodes of each depth.  All o' of a depth are w(l) or
    // 0, so the sums behind beta are w(l) times a count, exactly; the CAR
    // weights are made for every node at once and summed by a warp per depth.
    for (int n = 1 + tid; n < N; n += kEmThreads)
        sh.m.st[n] = exp(sh.m.st[n] - ordered_value(sh.cmax[depth[n] - 1]));
    __syncthreads();
    for (int l = 1 + warp; l <= maxd; l += kEmWarps) {
        double zs = 0.0;
        for (int n = 1 + lane; n < N; n += 32)
            if (depth[n] == l) zs += sh.m.st[n];
        zs = warp_sum(zs);
        if (lane == 0) sh.zs[l - 1] = zs;
    }
    __syncthreads();
    for (int n = 1 + tid; n < N; n += kEmThreads) {
        const int l = depth[n] - 1;
        const double op = sh.w[n][1];
        const double w = op != 0.0 ? op : (double)(float)(l < 64 ? P.wl[l] : pow(P.w_base, l + 1.0));
        const double d1 = w * sh.n0[l] - op, n1 = w * sh.n1[l] - op * sh.w[n][0];
        sh.w[n][2] = d1 > 0.0 ? (float)(n1 / d1) : 0.f;
        sh.w[n][3] = (float)(sh.m.st[n] / sh.zs[l]);
    }
    __syncthreads();
    // the objective (Eq. advance) and each proposal's gradient terms; the
    // nodes' first and last children
    double2 J = make_double2(0.0, 0.0);
    for (int n = tid; n < N; n += kEmThreads) {
        double st = 0.0, sz = 0.0;
        if (n) {
            const double ot = sh.w[n][0], op = sh.w[n][1];
            const double bz = (double)sh.w[n][2] * (double)sh.w[n][3];
            if (op != 0.0) {
                const double lqn = ot > 0.0 ? sh.lqt[n] : sh.lqz[n];
                J.x += op * (lqn - bz * sh.lqt[n]);
                st = op * (ot - bz);
                sz = op * (1.0 - ot);
            }
            const int a = par[n];
            int k = n - 1, m = n + 1;
            while (k > a && par[k] != a) --k;
            while (m < N && par[m] != a) ++m;
            sh.prev[n] = (short)(k > a ? k : 0);
            sh.next[n] = (short)(m < N ? m : 0);
            if (k <= a) sh.first[a] = (short)n;
            if (m >= N) sh.last[a] = (short)n;
        }
        sh.m.st[n] = st;
        sh.m.sz[n] = sz;
    }
    J = block_sum(J, sh.red);
    // subtree sums (the proposals whose path goes through a node)
    for (int l = maxd - 1; l >= 0; --l) {
        for (int a = tid; a < N; a += kEmThreads) {
            if (depth[a] != l || !sh.last[a]) continue;
            double st = sh.m.st[a], sz = sh.m.sz[a];
            for (int n = sh.last[a]; n; n = sh.prev[n]) {
                st += sh.m.st[n];
                sz += sh.m.sz[n];
            }
            sh.m.st[a] = st;
            sh.m.sz[a] = sz;
        }
        __syncthreads();
    }
    const double scale = Nb.x > 0.0 ? 1.0 / ((double)P.B * Nb.x * P.ts.Td) : 0.0;
    if (tid == 0) o.loss[b] = Nb.x > 0.0 ? (float)(-J.x / Nb.x) : 0.f;
    for (int x = tid; x < N; x += kEmThreads) {
        if (x) {
            TreeCoef cf;
            cf.t = __ldg(P.given_tokens + n0 + x);
            cf.ct = (float)(sh.m.st[x] * scale);
            cf.z = sh.z[x];
            cf.cz = (float)(sh.m.sz[x] * scale);
            if (cf.z == cf.t) {
                cf.ct = (float)((sh.m.st[x] + sh.m.sz[x]) * scale);
                cf.z = -1;
                cf.cz = 0.f;
            }
            P.tcoef[n0 + x] = cf;
        }
        float g = 0.f;  // the row's dense factor: its children's, in node order
        for (int n = sh.first[x]; n; n = sh.next[n])
            g += (float)((sh.m.st[n] + sh.m.sz[n]) * scale);
        P.tg[n0 + x] = g;
        if (o.corr_tokens) o.corr_tokens[n0 + x] = sh.z[x];
        if (o.weights)
            reinterpret_cast<float4*>(o.weights)[n0 + x] =
                x ? make_float4(sh.w[x][0], sh.w[x][1], sh.w[x][2], sh.w[x][3])
                  : make_float4(0.f, 0.f, 0.f, 0.f);
        if (o.logq_tok && x == 0) o.logq_tok[n0] = 0.f;
        if (o.logq_corr) o.logq_corr[n0 + x] = sh.lqzn[x];
        if (o.logkappa) o.logkappa[n0 + x] = (float)sh.lk[x];
        if (o.logkappa_corr) o.logkappa_corr[n0 + x] = (float)sh.lkc[x];
        if (o.logkappa_ref) o.logkappa_ref[n0 + x] = (float)sh.lkr[x];
    }
}

template <typename T>
__global__ void __launch_bounds__(kEmThreads) k_tree_em(Problem<T> P, vsd_tree_em_outputs o) {
    extern __shared__ __align__(128) unsigned char dsm[];
    TreeEmShared& sh = *reinterpret_cast<TreeEmShared*>(dsm);
    const int N = P.N, b = blockIdx.x, n0 = b * N;
    grid_launch_next();
    const bool ok = tree_load<kEmThreads>(P, b, sh.t);
    grid_wait();
    if (ok) {
        if (threadIdx.x == 0) P.tbad[b] = 0;
        tree_em_nodes<T>(P, o, b, sh);
    } else {
        for (int n = threadIdx.x; n < N; n += kEmThreads) {
            P.tcoef[n0 + n] = TreeCoef{-1, 0.f, -1, 0.f};
            P.tg[n0 + n] = 0.f;
            if (o.corr_tokens) o.corr_tokens[n0 + n] = -1;
            if (o.weights)
                reinterpret_cast<float4*>(o.weights)[n0 + n] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (threadIdx.x == 0) {
            atomicOr(P.status, VSD_STATUS_BAD_TREE);
            P.tbad[b] = 1;
            o.loss[b] = 0.f;
        }
    }
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) last = atomic_add_acq_rel(P.prefix_done, 1) == P.B - 1;
    __syncthreads();
    if (last && threadIdx.x < 32) loss_mean(o.loss, P.B, threadIdx.x);
}

// ------------------------------------------------------------ k_tree_grad
// Row r of the gradient: g q(v) minus the sparse terms of r's children.  The
// terms are merged by token in a fixed order (sorted by token, then by child)
// so that the sums do not depend on scheduling.  The dense part is written
// first, eight 16-byte vectors in flight per thread (a row without one is
// written as zeros and not read); then one thread per merged term writes its
// element.  What bounds it: the rows' reads and writes (64 trees of 60 nodes,
// V = 32000: 246 MB written, about half of the draft rows read).
struct TreeGradTerm {
    int tok, key;  // token; 2 n for node n's own token, 2 n + 1 for its corrected one
    float cf;
};
inline size_t tree_grad_smem_bytes(int N) { return (size_t)N * 4 * sizeof(TreeGradTerm); }

template <typename T, bool VEC, typename G>
__global__ void __launch_bounds__(kThreads) k_tree_grad(Problem<T> P, G* grad) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ int s_n;
    constexpr int PV = Traits<T>::kPerVec;
    const int N = P.N, r = blockIdx.x, b = r / N, u = r - b * N, n0 = b * N;
    TreeGradTerm* tm = reinterpret_cast<TreeGradTerm*>(dsm);  // [2 N] as gathered, then merged
    TreeGradTerm* srt = tm + 2 * N;                           // [2 N] sorted
    const int64_t V = P.V;
    G* g = grad + (int64_t)r * V;
    const T* x = P.draft + (int64_t)r * V;
    const int32_t* par = P.parent + (int64_t)n0;
    if (threadIdx.x == 0) s_n = 0;
    grid_wait();
    __syncthreads();
    const bool bad = ld_cg(P.tbad + b) != 0;
    if (!bad) {  // the children's terms
        for (int n = u + 1 + threadIdx.x; n < N; n += kThreads) {
            if (__ldg(par + n) != u) continue;
            const TreeCoef cf = ld_cg_rec(P.tcoef + n0 + n);
            const int slot = atomicAdd(&s_n, cf.z >= 0 ? 2 : 1);
            tm[slot] = TreeGradTerm{cf.t, 2 * n, cf.ct};
            if (cf.z >= 0) tm[slot + 1] = TreeGradTerm{cf.z, 2 * n + 1, cf.cz};
        }
    }
    const float gr = bad ? 0.f : ld_cg(P.tg + r);
    const RowRec rec = ld_cg(P.rows + r);
    __syncthreads();
    const int nt = s_n;
    const float gq = (nt == 0 && gr == 0.f) ? 0.f : gr * rec.izx;
    const float mx = rec.mx, c = P.ts.c;
    const bool dense = gq != 0.f && isfinite(mx);
    for (int i = threadIdx.x; i < nt; i += kThreads) {  // rank sort by (token, key)
        int rank = 0;
        for (int j = 0; j < nt; ++j)
            rank += tm[j].tok < tm[i].tok || (tm[j].tok == tm[i].tok && tm[j].key < tm[i].key);
        srt[rank] = tm[i];
    }
    // the terms' logits, before the row is written (the gradient may take the
    // draft's place)
    __syncthreads();
    if (dense)
        for (int i = threadIdx.x; i < nt; i += kThreads) {
            const int t = srt[i].tok;
            tm[i].cf = t >= 0 && t < V ? elem_value_cg(x, t) : 0.f;
        }
    __syncthreads();
    if constexpr (VEC) {
        constexpr int U = 8, NP = PV / 2;
        const uint64_t pol = policy_evict_first();
        const int nvec = (int)(V / PV);
        const uint64_t mx2 = f2(mx, mx), c2 = f2(c, c), gq2 = f2(gq, gq);
        for (int i0 = threadIdx.x; i0 < nvec; i0 += kThreads * U) {
            uint4 buf[U];
            if (dense) {
#pragma unroll
                for (int k = 0; k < U; ++k)
                    if (i0 + k * kThreads < nvec)
                        buf[k] = ld_stream(x + (int64_t)(i0 + k * kThreads) * PV, pol);
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const int i = i0 + k * kThreads;
                if (i >= nvec) break;
                float o[PV];
                if (dense) {
                    uint64_t pr[NP];
                    vec_pairs<T>(buf[k], pr);
#pragma unroll
                    for (int q = 0; q < NP; ++q)
                        f2split(f2mul(gq2, f2_mass(pr[q], mx2, c2)), o[2 * q], o[2 * q + 1]);
                } else {
#pragma unroll
                    for (int e = 0; e < PV; ++e) o[e] = 0.f;
                }
                grad_store<T, G, PV>(g, (int64_t)i * PV, o, pol);
            }
        }
    } else {
        for (int64_t v = threadIdx.x; v < V; v += kThreads) {
            const float val = dense ? gq * ex2((elem_value(x, v) - mx) * c) : 0.f;
            if constexpr (sizeof(G) == 2)
                g[v] = __float2bfloat16_rn(val);
            else
                g[v] = val;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nt; i += kThreads) {  // a token's first term sums them, in order
        const int t = srt[i].tok;
        if ((i && srt[i - 1].tok == t) || t < 0 || t >= V) continue;
        float cf = srt[i].cf;
        for (int j = i + 1; j < nt && srt[j].tok == t; ++j) cf += srt[j].cf;
        const float val = (dense ? gq * ex2((tm[i].cf - mx) * c) : 0.f) - cf;
        if constexpr (sizeof(G) == 2)
            g[t] = __float2bfloat16_rn(val);
        else
            g[t] = val;
    }
}

// ------------------------------------------------------------ sequential rule
// The sequential sibling rule (lossless multi-draft) at a node u with children
// c_1 .. c_m (node order): child i is accepted with probability
// min(1, p_i(t_i)/q_i(t_i)); after a rejection p_{i+1} = norm(max(0, p_i - q_i))
// (p_i kept if that has no mass) and q_{i+1} = q_i without t_i, renormalised.
//
// Which child of u is accepted first, and the correction token if none is,
// depend on u's row, its children and their uniforms alone, so every row is
// decided where it is read (k_tree_seq_rows, one block per row); the walk
// along the accepted path then only follows the rows' decisions (k_tree_seq).
//
// Every q_i is the same q but for a factor 1/Q_i (Q_i: the draft mass not yet
// removed), and max(0, max(0, p - a q) - b q) = max(0, p - (a + b) q) for
// a, b >= 0, so with p_i = P_i / T_i
//   P_i(v) = max(0, p(v) - A_i q(v)),  A_{i+1} = A_i + T_i / Q_i,  T_i = sum P_i
// and a removed token keeps the A of the step that removed it.  Each rejected
// child therefore costs one read of the row (from L2, where the row pass left
// it) with one multiply-add more than the plain residual, however many
// siblings went before it.
struct SeqCtl {
    int m;          // children of the row's node
    int next;       // the accepted child (node index), -1 so far
    int out;        // the correction token
    double A, T, Q; // A_i, T_i, Q_i of the child tried next
    double An;      // A_{i+1}
    float ah, al;   // A_{i+1} in two floats
};
// Per child of the row's node, in node order (dynamic shared memory, sized by
// the tree's nodes).
struct SeqKids {
    double* p;      // p and q of its token at the row
    double* q;
    float2* A;      // the A its token keeps once removed, in two floats
    int* tok;
    int* kid;       // its node
    float* ua;      // its uniforms
    float* uc;
};
inline size_t seq_smem_bytes(int N) { return (size_t)N * 40; }
__device__ __forceinline__ SeqKids seq_kids(unsigned char* base, int N) {
    SeqKids s;
    s.p = reinterpret_cast<double*>(base);
    s.q = s.p + N;
    s.A = reinterpret_cast<float2*>(s.q + N);
    s.tok = reinterpret_cast<int*>(s.A + N);
    s.kid = s.tok + N;
    s.ua = reinterpret_cast<float*>(s.kid + N);
    s.uc = s.ua + N;
    return s;
}

__device__ __forceinline__ float2 two_floats(double a) {
    const float h = (float)a;
    return make_float2(h, (float)(a - (double)h));
}
// max(0, p - A q) from A in two floats (48 of the double's 53 bits); each product
// is exact inside its multiply-add, the difference rounded to float twice.
__device__ __forceinline__ float seq_mass(float p, float q, float ah, float al) {
    return fmaxf(fmaf(-al, q, fmaf(-ah, q, p)), 0.f);
}

// The masses of one row after some rejections: A for every token but the
// first `nrem` children's, which keep their own.
struct SeqMass {
    MassRes mr;
    float ah, al;
    const int* tok;
    const float2* A;
    int nrem;
    // (the first of equal tokens is the one that was removed)
    __device__ float operator()(float fx, float fy, int v) const {
        const float p = ex2((fy - mr.my) * mr.c) * mr.izy;
        const float q = ex2((fx - mr.mx) * mr.c) * mr.izx;
        for (int j = 0; j < nrem; ++j)
            if (tok[j] == v) return seq_mass(p, q, A[j].x, A[j].y);
        return seq_mass(p, q, ah, al);
    }
};

// Sum of the masses of one chunk (warp).
template <typename T>
__device__ __forceinline__ float seq_chunk(const uint4 (&bx)[kLoads], const uint4 (&by)[kLoads],
                                           int ch, const SeqMass& sm, int lane) {
    constexpr int PV = Traits<T>::kPerVec, NP = PV / 2, CE = chunk_elems<T>();
    bool some = false;  // a removed token lies in this chunk
    for (int j = lane; j < sm.nrem; j += 32) some |= (unsigned)(sm.tok[j] - ch * CE) < (unsigned)CE;
    float acc = 0.f;
    if (__any_sync(0xffffffffu, some)) {
#pragma unroll
        for (int k = 0; k < kLoads; ++k) {
            float fx[PV], fy[PV];
            unpack<T>(bx[k], fx);
            unpack<T>(by[k], fy);
#pragma unroll
            for (int e = 0; e < PV; ++e)
                acc += sm(fx[e], fy[e], ch * CE + k * 32 * PV + lane * PV + e);
        }
        return warp_sum(acc);
    }
    const MassRes& mr = sm.mr;
    const uint64_t mx2 = f2(mr.mx, mr.mx), my2 = f2(mr.my, mr.my), c2 = f2(mr.c, mr.c);
    const uint64_t izx2 = f2(mr.izx, mr.izx), izy2 = f2(mr.izy, mr.izy);
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
        uint64_t px[NP], py[NP];
        vec_pairs<T>(bx[k], px);
        vec_pairs<T>(by[k], py);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            float q0, q1, p0, p1;
            f2split(f2mul(f2_mass(px[i], mx2, c2), izx2), q0, q1);
            f2split(f2mul(f2_mass(py[i], my2, c2), izy2), p0, p1);
            acc += seq_mass(p0, q0, sm.ah, sm.al) + seq_mass(p1, q1, sm.ah, sm.al);
        }
    }
    return warp_sum(acc);
}

// One read of row r: tab[ch].y = the chunk sums of its masses (block).
template <typename T, bool VEC, int S>
__device__ void seq_stream(const Problem<T>& P, int r, Ring<S>* rg, float4* tab, const SeqMass& sm) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t V = P.V;
    const T* x = P.draft + (int64_t)r * V;
    const T* y = P.target + (int64_t)r * V;
    const uint64_t pol = policy_evict_normal();
    if constexpr (VEC) {
        ring_stream<T, true>(rg, x, y, V, 0, P.nch, pol, pol, P.status,
                             [&](int ch, const uint4 (&bx)[kLoads], const uint4 (&by)[kLoads]) {
                                 const float t = seq_chunk<T>(bx, by, ch, sm, lane);
                                 if (lane == 0) tab[ch] = make_float4(0.f, t, 0.f, 0.f);
                             });
    } else {
        for (int ch = warp; ch < P.nch; ch += kWarps) {
            uint4 bx[kLoads], by[kLoads];
            load_chunk<T, VEC>(x, V, ch, lane, pol, bx);
            load_chunk<T, VEC>(y, V, ch, lane, pol, by);
            const float t = seq_chunk<T>(bx, by, ch, sm, lane);
            if (lane == 0) tab[ch] = make_float4(0.f, t, 0.f, 0.f);
        }
    }
    __syncthreads();
}

// Inverse-CDF draw from the masses whose chunk sums are in tab (warp; -1 if
// there is no mass).
template <typename T, bool VEC>
__device__ int seq_draw(const Problem<T>& P, int r, const float4* tab, const TableSum& S, float u,
                        const SeqMass& sm, int lane, uint4* buf) {
    const Located loc = table_locate(tab, P.nch, 0, 0.f, P.ts.c, S, u, lane);
    if (loc.ch < 0) return -1;
    return warp_rescan<T, VEC, true, true>(P.draft + (int64_t)r * P.V, P.target + (int64_t)r * P.V,
                                           P.V, loc.ch, loc.tc, sm, lane, policy_evict_normal(), buf);
}

// The decision at node u = row r (block, after the row's pass): tries its
// children in turn.  Per tried child tnode[].lq = alpha, .acc, .zp = 1 (0 for
// the others), for every child .la; tlist[r] = the accepted child, 0 if u has
// no children, -1 if all were rejected, with the correction token in
// es.corr[r].
template <typename T, bool VEC, int S>
__device__ void tree_seq_row(const Problem<T>& P, int r, Ring<S>* rg, float4* tab, SeqCtl& ct,
                             const SeqKids& s) {
    const int N = P.N, b = r / N, u = r - b * N, n0 = b * N;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t V = P.V;
    const int32_t* par = P.parent + (int64_t)n0;
    const float c = P.ts.c;
    const RowRec rec = ld_cg(P.rows + r);
    if (warp == 0) {  // the children, in node order
        int m = 0;
        for (int g = u + 1; g < N; g += 32) {
            const bool is = g + lane < N && __ldg(par + g + lane) == u;
            const unsigned bal = __ballot_sync(0xffffffffu, is);
            if (is) s.kid[m + __popc(bal & ((1u << lane) - 1u))] = g + lane;
            m += __popc(bal);
        }
        if (lane == 0) {
            ct.m = m;
            ct.next = m ? -1 : 0;
            ct.out = -1;
            ct.A = 0.0;
            ct.T = ct.Q = 1.0;
        }
    }
    __syncthreads();
    const int m = ct.m;
    if (threadIdx.x == 0 && rec.flags && (m || P.tout.row_stats))
        atomicOr(P.status, VSD_STATUS_BAD_ROW);
    for (int i = threadIdx.x; i < m; i += kThreads) {
        const int n = n0 + s.kid[i], tok = __ldg(P.given_tokens + n);
        TreeNodeRec nr;
        nr.la = -INFINITY;
        nr.lq = 0.f;
        nr.acc = nr.zp = 0;
        nr.lq_zp = nr.la_zp = nr.lq_zr = nr.la_zr = 0.f;
        nr.zr = -1;
        nr.pad[0] = nr.pad[1] = nr.pad[2] = 0;
        double p = 0.0, q = 0.0;
        if (tok < 0 || tok >= V) {
            atomicOr(P.status, VSD_STATUS_BAD_TOKEN);
        } else if (!rec.flags) {
            const float xv = elem_value(P.draft + (int64_t)r * V, tok);
            const float yv = elem_value(P.target + (int64_t)r * V, tok);
            float lq;
            token_logs_vals(xv, yv, rec, P.ts.invTd, &lq, &nr.la);
            p = exp(((double)yv - rec.my) * P.ts.invTd - rec.lzy);
            q = exp(((double)xv - rec.mx) * P.ts.invTd - rec.lzx);
        }
        s.ua[i] = __ldg(P.u_accept + n);
        s.uc[i] = __ldg(P.u_correct + n);
        s.tok[i] = tok;
        s.p[i] = p;
        s.q[i] = q;
        P.tnode[n] = nr;
    }
    __syncthreads();
    const MassRes mr{rec.mx, rec.my, rec.izx, rec.izy, c};
    for (int i = 0; i < m; ++i) {
        if (warp == 0) {
            const int n = n0 + s.kid[i], t = s.tok[i];
            int before = -1;  // the earlier sibling that removed t, if any
            for (int j = 0; j < i && before < 0; ++j)
                if (s.tok[j] == t) before = j;
            const double Q = ct.Q, A = ct.A, Tm = ct.T;
            const double At = before >= 0 ? (double)s.A[before].x + (double)s.A[before].y : A;
            // p_i, q_i at t, and A's step T_i / Q_i: three quotients on three lanes
            const double num = lane == 0 ? fmax(0.0, s.p[i] - At * s.q[i]) : lane == 1 ? s.q[i] : Tm;
            const double den = lane == 0 ? Tm : Q;
            const double quo = den > 0.0 ? num / den : 0.0;
            const double pi = __shfl_sync(0xffffffffu, quo, 0);
            const double qi = before >= 0 ? 0.0 : __shfl_sync(0xffffffffu, quo, 1);
            const double step = __shfl_sync(0xffffffffu, quo, 2);
            double alpha = 0.0;
            if (!rec.flags && t >= 0 && t < V)
                alpha = qi > 0.0 ? fmin(1.0, pi / qi) : (pi > 0.0 ? 1.0 : 0.0);
            const bool a = s.ua[i] <= alpha && !rec.flags;
            if (lane == 0) {
                P.tnode[n].lq = (float)alpha;
                P.tnode[n].acc = a ? 1 : 0;
                P.tnode[n].zp = 1;
                if (a) ct.next = s.kid[i];
                ct.An = A + step;
                const float2 h = two_floats(ct.An);
                ct.ah = h.x;
                ct.al = h.y;
                if (before < 0) ct.Q = Q - s.q[i];
            }
        }
        __syncthreads();
        if (ct.next > 0) break;
        if (!rec.flags) {
            // T_{i+1} (one read of the row); the draw after the last rejection
            const float uc = s.uc[i];
            const SeqMass sm{mr, ct.ah, ct.al, s.tok, s.A, i};
            seq_stream<T, VEC>(P, r, rg, tab, sm);
            if (warp == 0) {
                const TableSum Rt = table_sum(tab, P.nch, 0, 0.f, c, lane);
                // (no mass left: p_i is kept, and the draw is from it)
                const int tok = i < m - 1 ? -1
                                : Rt.Z > 0.0 ? seq_draw<T, VEC>(P, r, tab, Rt, uc, sm, lane, warp_chunks(rg))
                                             : -2;
                if (lane == 0) {
                    if (Rt.Z > 0.0 && Rt.Z < INFINITY) {
                        ct.A = ct.An;
                        ct.T = Rt.Z;
                    }
                    s.A[i] = two_floats(ct.A);
                    ct.out = tok;
                }
            }
            __syncthreads();
            if (ct.out == -2) {
                const float2 h = two_floats(ct.A);
                const SeqMass keep{mr, h.x, h.y, s.tok, s.A, i};
                __syncthreads();
                seq_stream<T, VEC>(P, r, rg, tab, keep);
                if (warp == 0) {
                    const TableSum Pt = table_sum(tab, P.nch, 0, 0.f, c, lane);
                    const int tok =
                        Pt.Z > 0.0 ? seq_draw<T, VEC>(P, r, tab, Pt, uc, keep, lane,
                                                         warp_chunks(rg)) : -1;
                    if (lane == 0) ct.out = tok;
                }
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        P.tlist[r] = ct.next;
        P.es.corr[r] = ct.out;
    }
}

// One block per node row.  A leaf's row is read for the statistics output, and
// where the rows are few (read_leaves), since it costs nothing beside the others
// then; else the row a bonus token needs is read by k_tree_seq.
// What bounds it: the row reads and row tails (3840 rows of 2 x 64 KB), and
// the reads after a rejection, which come from L2.  64 trees of 60 nodes,
// V = 32000: 210 to 225 us a call; 5.46 ms with the rule run along the path by one
// block per tree, in an fp64 recursion per element over the earlier siblings.
template <typename T, bool VEC, int S>
__global__ void __launch_bounds__(kThreads, VEC ? kRowBlocks : 1) k_tree_seq_rows(Problem<T> P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ RowShared sh;
    __shared__ SeqCtl ct;
    Ring<S>* rg;
    float4* tab;
    smem_views<VEC>(dsm, rg, tab, P.timeout_ns, P.hold_copies != 0);
    grid_launch_next();
    const SeqKids kids = seq_kids(reinterpret_cast<unsigned char*>(tab + P.nch), P.N);
    const int r = blockIdx.x, N = P.N, b = r / N, u = r - b * N;
    int has = 0;
    for (int n = u + 1 + threadIdx.x; n < N && !has; n += kThreads)
        has = __ldg(P.parent + (int64_t)b * N + n) == u;
    has = __syncthreads_or(has);
    if (!has && !P.tout.row_stats && !P.read_leaves) {
        grid_wait();
        if (threadIdx.x == 0) P.tlist[r] = 0;
        return;
    }
    // (a leaf's draw from p may become the bonus token; a leaf read for that alone
    // sets no status bit here)
    row_pass<T, VEC, true, kNoToken, false, true>(P, r, rg, tab, sh, !has);
    __syncthreads();
    if (threadIdx.x == 0 && P.tout.row_stats)
        reinterpret_cast<float4*>(P.tout.row_stats)[r] = ld_cg(P.rstats + r);
    tree_seq_row<T, VEC>(P, r, rg, tab, ct, kids);
}

struct TreeSeqShared {
    TreeShared2 t;
    double lk[1024];
    float la[1024];
    int next[1024];
    unsigned char on[1024];  // on the accepted path
    int best, lastkid;
};

// One block per tree: the accepted path, and every node's outputs.
template <typename T, bool VEC, int S>
__global__ void __launch_bounds__(kThreads) k_tree_seq(Problem<T> P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ RowShared rsh;
    Ring<S>* rg;
    float4* tab;
    smem_views<VEC>(dsm, rg, tab, P.timeout_ns, P.hold_copies != 0);
    TreeSeqShared& sh = *reinterpret_cast<TreeSeqShared*>(tab + P.nch);
    grid_wait();
    const int N = P.N, b = blockIdx.x, n0 = b * N;
    const vsd_tree_outputs& o = P.tout;
    if (!tree_load<kThreads>(P, b, sh.t)) {
        for (int n = threadIdx.x; n < N; n += kThreads) {
            o.alpha[n0 + n] = 0.f;
            o.accept[n0 + n] = 0;
            o.path_accept[n0 + n] = 0;
            o.logkappa[n0 + n] = -INFINITY;
            o.corr_tokens[n0 + n] = -1;
        }
        if (threadIdx.x == 0) {
            atomicOr(P.status, VSD_STATUS_BAD_TREE);
            o.deepest[b] = -1;
            o.accept_len[b] = -1;
            o.bonus[b] = -1;
        }
        return;
    }
    for (int n = threadIdx.x; n < N; n += kThreads) {
        sh.next[n] = P.tlist[n0 + n];
        sh.la[n] = n ? P.tnode[n0 + n].la : 0.f;
        sh.on[n] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int u = 0;
        sh.on[0] = 1;
        while (sh.next[u] > 0) {  // (a child comes after its parent)
            u = sh.next[u];
            sh.on[u] = 1;
        }
        sh.best = u;
        sh.lastkid = 0;
        sh.lk[0] = 0.0;
    }
    // log kappa: the path validity (Eq. 2) of every node, level by level
    for (int l = 1; l <= sh.t.maxd; ++l) {
        __syncthreads();
        for (int n = threadIdx.x; n < N; n += kThreads)
            if (sh.t.depth[n] == l) sh.lk[n] = sh.lk[sh.t.par[n]] + (double)sh.la[n];
    }
    __syncthreads();
    const int best = sh.best;
    for (int n = threadIdx.x; n < N; n += kThreads) {
        const int pn = n ? sh.t.par[n] : 0;
        float alpha = n ? 0.f : 1.f;
        int acc = n ? 0 : 1;
        if (n && sh.on[pn] && P.tnode[n0 + n].zp) {  // tried
            alpha = P.tnode[n0 + n].lq;
            acc = P.tnode[n0 + n].acc;
        }
        o.alpha[n0 + n] = alpha;
        o.accept[n0 + n] = acc ? 1 : 0;
        o.path_accept[n0 + n] = sh.on[n];
        o.logkappa[n0 + n] = (float)sh.lk[n];
        o.corr_tokens[n0 + n] = -1;
        if (n && pn == best) atomicMax(&sh.lastkid, n);
    }
    __syncthreads();
    const bool leaf = sh.lastkid == 0;
    if (leaf && !P.tout.row_stats && !P.read_leaves) {  // the leaf's row, for the bonus token
        row_pass<T, VEC, true, kNoToken, false>(P, n0 + best, rg, tab, rsh);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        o.deepest[b] = best;
        o.accept_len[b] = sh.t.depth[best];
        const int tok = leaf ? ld_cg(P.rows + n0 + best).ps : P.es.corr[n0 + best];
        if (leaf && ld_cg(P.rows + n0 + best).flags) atomicOr(P.status, VSD_STATUS_BAD_ROW);
        if (!leaf) o.corr_tokens[n0 + sh.lastkid] = tok;
        o.bonus[b] = tok;
    }
}

}  // namespace vsd
