// vsd_tree.cuh -- draft trees beyond independent branch verification (App. E
// trees): the E-step + M-step with every node a latent proposal, and tree
// verification with the sequential sibling rule (lossless multi-draft).
//
//   k_tree_rows  one block per node row u: the row pass (tables, statistics,
//                the target's argmax, a draw from p with u's uniform), then
//                for every child x of u its token's test at u's row (Eq. 1,
//                each branch alone) and, for the EM, the draws a corrected
//                path may take at x: from p with x's uniform (below a
//                rejection) and from the residual norm(max(0, p - q)) (the
//                first rejection; one more read of the row when a child is
//                rejected).
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
    int zp;        // draw from p at the parent's row with x's u_correct
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

// ------------------------------------------------------------ k_tree_rows
template <typename T, bool VEC>
__device__ void tree_row_children(const Problem<T>& P, int r, Ring* rg, float4* tab, int* s_any) {
    const int N = P.N;
    const int64_t V = P.V;
    const int b = r / N, u = r - b * N, n0 = b * N;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t* par = P.parent + (int64_t)n0;
    const T* x = P.draft + (int64_t)r * V;
    const T* y = P.target + (int64_t)r * V;
    const float c = P.ts.c;
    const uint64_t pol = policy_evict_normal();
    const RowRec rec = ld_cg(P.rows + r);
    if (threadIdx.x == 0) *s_any = 0;
    __syncthreads();
    // the target's table for the draws from p (each warp, identical values)
    float My = 0.f;
    TableSum Sy{0, 0, 0.0};
    My = table_max(tab, P.nch, 1, lane);
    Sy = table_sum(tab, P.nch, 1, frame_of(My), c, lane);
    int k = 0;
    for (int n = u + 1; n < N; ++n) {
        if (__ldg(par + n) != u) continue;
        if (k++ % kWarps != warp) continue;
        TreeNodeRec nr;
        nr.la = -INFINITY;
        nr.lq = -INFINITY;
        nr.zp = -1;
        nr.lq_zp = nr.la_zp = -INFINITY;
        nr.zr = -1;
        nr.lq_zr = nr.la_zr = -INFINITY;
        nr.pad[0] = nr.pad[1] = nr.pad[2] = 0;
        const int tok = __ldg(P.given_tokens + n0 + n);
        if (tok < 0 || tok >= V) {
            if (lane == 0) atomicOr(P.status, VSD_STATUS_BAD_TOKEN);
        } else if (!rec.flags) {
            token_logs(x, y, tok, rec, P.ts.invTd, &nr.lq, &nr.la);
        }
        nr.acc = nr.la > -INFINITY && __ldg(P.u_accept + n0 + n) <= expf(nr.la);
        if (!rec.flags) {
            int zp = warp_sample<T, VEC>(x, y, V, tab, P.nch, 1, My, Sy,
                                         __ldg(P.u_correct + n0 + n), c, lane, pol);
            if (zp >= V) zp = -1;
            nr.zp = zp;
            if (zp >= 0) token_logs(x, y, zp, rec, P.ts.invTd, &nr.lq_zp, &nr.la_zp);
        }
        if (lane == 0) {
            P.tnode[n0 + n] = nr;
            if (!nr.acc) *s_any = 1;
        }
    }
    __syncthreads();
    if (!*s_any || rec.flags) return;
    // a child is rejected: the residual max(0, p - q) of the row, and each
    // rejected child's draw from it (or from p if it has no mass)
    const MassRes mr{rec.mx, rec.my, rec.izx, rec.izy, c};
    stream_residual<T, VEC>(rg, x, y, V, 0, P.nch, tab, mr, P.status);
    __syncthreads();
    const TableSum Rt = table_sum(tab, P.nch, 0, 0.f, c, lane);
    k = 0;
    for (int n = u + 1; n < N; ++n) {
        if (__ldg(par + n) != u) continue;
        if (k++ % kWarps != warp) continue;
        TreeNodeRec nr = P.tnode[n0 + n];  // written by this warp above
        if (nr.acc) continue;
        int zr = -1;
        if (Rt.Z > 0.0) {
            const Located loc =
                table_locate(tab, P.nch, 0, 0.f, c, Rt, __ldg(P.u_correct + n0 + n), lane);
            if (loc.ch >= 0)
                zr = warp_rescan<T, VEC, true, true>(x, y, V, loc.ch, loc.tc, mr, lane, pol);
            if (zr >= V) zr = -1;
        } else {
            zr = nr.zp;  // no residual mass: the draw from p with the same uniform
        }
        nr.zr = zr;
        if (zr >= 0) token_logs(x, y, zr, rec, P.ts.invTd, &nr.lq_zr, &nr.la_zr);
        if (lane == 0) P.tnode[n0 + n] = nr;
    }
}

template <typename T, bool VEC>
__global__ void __launch_bounds__(kThreads) k_tree_rows(Problem<T> P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ RowShared sh;
    __shared__ int s_any;
    Ring* rg = nullptr;
    float4* tab;
    if (VEC) {
        rg = reinterpret_cast<Ring*>(dsm);
        tab = reinterpret_cast<float4*>(dsm + sizeof(Ring));
        ring_init(rg, P.timeout_ns);
    } else {
        tab = reinterpret_cast<float4*>(dsm);
    }
    const int r = blockIdx.x;
    row_pass<T, VEC, true, kNoToken, true>(P, r, rg, tab, sh);
    __syncthreads();
    tree_row_children<T, VEC>(P, r, rg, tab, &s_any);
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
template <typename T>
__device__ bool tree_load(const Problem<T>& P, int b, TreeShared2& sh) {
    const int N = P.N;
    const int32_t* par = P.parent + (int64_t)b * N;
    int badl = 0;
    for (int n = threadIdx.x; n < N; n += kThreads) {
        const int pn = __ldg(par + n);
        sh.par[n] = pn;
        badl |= n == 0 ? pn != -1 : (pn < 0 || pn >= n);
    }
    const int bad = __syncthreads_or(badl);
    if (bad) return false;
    // depths by pointer doubling: depth[n] steps from n to anc[n]
    for (int n = threadIdx.x; n < N; n += kThreads) {
        sh.depth[n] = n ? 1 : 0;
        sh.anc[n] = (short)(n ? sh.par[n] : 0);
    }
    if (threadIdx.x == 0) sh.maxd = 0;
    for (;;) {
        __syncthreads();
        short a[1024 / kThreads];
        int d[1024 / kThreads];
        int more = 0;
#pragma unroll
        for (int k = 0; k < 1024 / kThreads; ++k) {
            const int n = threadIdx.x + k * kThreads;
            if (n >= N) break;
            a[k] = sh.anc[sh.anc[n]];
            d[k] = sh.depth[n] + sh.depth[sh.anc[n]];
            more |= a[k] != 0;
        }
        more = __syncthreads_or(more);
#pragma unroll
        for (int k = 0; k < 1024 / kThreads; ++k) {
            const int n = threadIdx.x + k * kThreads;
            if (n >= N) break;
            sh.anc[n] = a[k];
            sh.depth[n] = d[k];
        }
        if (!more) break;
    }
    __syncthreads();
    int md = 0;
    for (int n = threadIdx.x; n < N; n += kThreads) md = max(md, sh.depth[n]);
    atomicMax(&sh.maxd, md);
    __syncthreads();
    return true;
}

// ------------------------------------------------------------ k_tree_em
// The M-step of one tree, in double precision on one thread (a tree has at
// most 1024 nodes; the arithmetic follows the proposals in node order, so the
// result does not depend on scheduling).  Scratch per node in shared memory.
struct TreeEmShared {
    TreeShared2 t;
    double lk[1024], lkc[1024], lkr[1024], lqt[1024], lqz[1024];
    double st[1024], sz[1024];   // subtree sums of the gradient terms
    float w[1024][4];            // o~, o', beta, zeta
    float lqzn[1024];            // log q of z'_x at its parent's row
    int z[1024];                 // corrected token z'_x
};

template <typename T>
__global__ void __launch_bounds__(kThreads) k_tree_em(Problem<T> P, vsd_tree_em_outputs o) {
    extern __shared__ __align__(128) unsigned char dsm[];
    TreeEmShared& sh = *reinterpret_cast<TreeEmShared*>(dsm);
    const int N = P.N, b = blockIdx.x, n0 = b * N;
    const bool ok = tree_load<T>(P, b, sh.t);
    if (!ok) {
        for (int n = threadIdx.x; n < N; n += kThreads) {
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
    } else if (threadIdx.x == 0) {
        P.tbad[b] = 0;
        const int* par = sh.t.par;
        const int* depth = sh.t.depth;
        // the E-step per node (R15): accepted paths, z', the sums along the paths
        sh.t.pacc[0] = 1;
        sh.lk[0] = sh.lkc[0] = sh.lkr[0] = sh.lqt[0] = sh.lqz[0] = 0.0;
        sh.z[0] = -1;
        sh.lqzn[0] = 0.f;
        for (int x = 1; x < N; ++x) {
            const int a = par[x];
            const TreeNodeRec nr = ld_cg_rec(P.tnode + n0 + x);
            const RowRec ra = ld_cg(P.rows + n0 + a);
            const int tok = __ldg(P.given_tokens + n0 + x);
            const bool pa = nr.acc && sh.t.pacc[a];
            sh.t.pacc[x] = pa;
            int zc;
            float lqz, laz;
            if (pa) {
                zc = tok; lqz = nr.lq; laz = nr.la;
            } else if (sh.t.pacc[a]) {  // the first rejection on the path: the residual
                zc = nr.zr; lqz = nr.lq_zr; laz = nr.la_zr;
            } else {                    // below a rejection: the draw from p
                zc = nr.zp; lqz = nr.lq_zp; laz = nr.la_zp;
            }
            if (zc < 0) { lqz = -INFINITY; laz = -INFINITY; }
            sh.z[x] = zc;
            sh.lqzn[x] = lqz;
            const double lar = (ra.flags || ra.ref < 0) ? -INFINITY : (double)ra.la_ref;
            sh.lk[x] = sh.lk[a] + (double)nr.la;
            sh.lkc[x] = sh.lkc[a] + (double)laz;
            sh.lkr[x] = sh.lkr[a] + lar;
            sh.lqt[x] = sh.lqt[a] + (double)nr.lq;
            sh.lqz[x] = sh.lqz[a] + (double)lqz;
        }
        // o~, o' (Algorithm 2 with w(depth))
        double Nb = 0.0;
        for (int n = 1; n < N; ++n) {
            // w(l) = w_base^l at the node's depth (trees may be deeper than the
            // host's table of w)
            const double wl = pow(P.w_base, (double)depth[n]);
            const bool ot = sh.lk[n] >= sh.lkr[n];
            const bool op = ot || sh.lkc[n] >= sh.lkr[n];
            sh.w[n][0] = ot ? 1.f : 0.f;
            sh.w[n][1] = op ? (float)wl : 0.f;
            Nb += op ? wl : 0.0;
        }
        // beta (leave-one-out) and zeta (softmax of q(z~)/tau, or log q in
        // zeta_mode 1) over the nodes of each depth
        for (int l = 1; l <= sh.t.maxd; ++l) {
            double num = 0.0, den = 0.0, cmax = -INFINITY;
            for (int n = 1; n < N; ++n) {
                if (depth[n] != l) continue;
                const double op = sh.w[n][1];
                num += op * sh.w[n][0];
                den += op;
                const double cq = (P.zeta_mode == 0 ? exp(sh.lqt[n]) : sh.lqt[n]) * P.inv_tau;
                cmax = fmax(cmax, cq);
            }
            double zs = 0.0;
            for (int n = 1; n < N; ++n) {
                if (depth[n] != l) continue;
                const double cq = (P.zeta_mode == 0 ? exp(sh.lqt[n]) : sh.lqt[n]) * P.inv_tau;
                zs += exp(cq - cmax);
            }
            for (int n = 1; n < N; ++n) {
                if (depth[n] != l) continue;
                const double op = sh.w[n][1];
                const double d1 = den - op, n1 = num - op * sh.w[n][0];
                sh.w[n][2] = d1 > 0.0 ? (float)(n1 / d1) : 0.f;
                const double cq = (P.zeta_mode == 0 ? exp(sh.lqt[n]) : sh.lqt[n]) * P.inv_tau;
                sh.w[n][3] = (float)(exp(cq - cmax) / zs);
            }
        }
        // the objective (Eq. advance), each proposal's terms, subtree sums
        // (the proposals whose path goes through a node)
        double J = 0.0;
        for (int n = 0; n < N; ++n) sh.st[n] = sh.sz[n] = 0.0;
        for (int n = 1; n < N; ++n) {
            const double ot = sh.w[n][0], op = sh.w[n][1];
            const double bz = (double)sh.w[n][2] * (double)sh.w[n][3];
            if (op == 0.0) continue;
            const double lqn = ot > 0.0 ? sh.lqt[n] : sh.lqz[n];
            J += op * (lqn - bz * sh.lqt[n]);
            sh.st[n] += op * (ot - bz);
            sh.sz[n] += op * (1.0 - ot);
        }
        for (int n = N - 1; n >= 1; --n) {  // children come after their parents
            sh.st[par[n]] += sh.st[n];
            sh.sz[par[n]] += sh.sz[n];
        }
        const double scale = Nb > 0.0 ? 1.0 / ((double)P.B * Nb * P.ts.Td) : 0.0;
        for (int n = 0; n < N; ++n) P.tg[n0 + n] = 0.f;
        o.loss[b] = Nb > 0.0 ? (float)(-J / Nb) : 0.f;
        for (int x = 1; x < N; ++x) {
            TreeCoef cf;
            cf.t = __ldg(P.given_tokens + n0 + x);
            cf.ct = (float)(sh.st[x] * scale);
            cf.z = sh.z[x];
            cf.cz = (float)(sh.sz[x] * scale);
            if (cf.z == cf.t) {
                cf.ct = (float)((sh.st[x] + sh.sz[x]) * scale);
                cf.z = -1;
                cf.cz = 0.f;
            }
            P.tcoef[n0 + x] = cf;
            P.tg[n0 + par[x]] += (float)((sh.st[x] + sh.sz[x]) * scale);
        }
    }
    __syncthreads();
    if (ok) {
        for (int n = threadIdx.x; n < N; n += kThreads) {
            if (o.corr_tokens) o.corr_tokens[n0 + n] = sh.z[n];
            if (o.weights)
                reinterpret_cast<float4*>(o.weights)[n0 + n] =
                    n ? make_float4(sh.w[n][0], sh.w[n][1], sh.w[n][2], sh.w[n][3])
                      : make_float4(0.f, 0.f, 0.f, 0.f);
            if (o.logq_tok) o.logq_tok[n0 + n] = n ? ld_cg(&P.tnode[n0 + n].lq) : 0.f;
            if (o.logq_corr) o.logq_corr[n0 + n] = sh.lqzn[n];
            if (o.logkappa) o.logkappa[n0 + n] = (float)sh.lk[n];
            if (o.logkappa_corr) o.logkappa_corr[n0 + n] = (float)sh.lkc[n];
            if (o.logkappa_ref) o.logkappa_ref[n0 + n] = (float)sh.lkr[n];
        }
    }
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(P.prefix_done, 1) == P.B - 1) {
            __threadfence();
            loss_mean(o.loss, P.B);
        }
    }
}

// ------------------------------------------------------------ k_tree_grad
// Row r of the gradient: g q(v) minus the sparse terms of r's children.  The
// terms are merged by token in a fixed order (sorted by token, then by child)
// so that the sums do not depend on scheduling.
constexpr int kTreeMaxTerms = 2048;
struct TreeGradShared {
    int tok[kTreeMaxTerms];
    float cf[kTreeMaxTerms];
    int skey[kTreeMaxTerms];
    float scf[kTreeMaxTerms];
    int n, nu;
};

template <typename T, bool VEC, typename G>
__global__ void __launch_bounds__(kThreads) k_tree_grad(Problem<T> P, G* grad) {
    __shared__ TreeGradShared sh;
    constexpr int PV = Traits<T>::kPerVec;
    const int N = P.N, r = blockIdx.x, b = r / N, u = r - b * N, n0 = b * N;
    const int64_t V = P.V;
    G* g = grad + (int64_t)r * V;
    const T* x = P.draft + (int64_t)r * V;
    const int32_t* par = P.parent + (int64_t)n0;
    if (threadIdx.x == 0) sh.n = 0;
    __syncthreads();
    const bool bad = ld_cg(P.tbad + b) != 0;
    if (!bad) {  // the children's terms
        for (int n = u + 1 + threadIdx.x; n < N; n += kThreads) {
            if (__ldg(par + n) != u) continue;
            const TreeCoef cf = ld_cg_rec(P.tcoef + n0 + n);
            const int slot = atomicAdd(&sh.n, cf.z >= 0 ? 2 : 1);
            // (order fixed below by the sort key: token, then child index)
            sh.tok[slot] = cf.t;
            sh.cf[slot] = cf.ct;
            sh.skey[slot] = 2 * n;
            if (cf.z >= 0) {
                sh.tok[slot + 1] = cf.z;
                sh.cf[slot + 1] = cf.cz;
                sh.skey[slot + 1] = 2 * n + 1;
            }
        }
    }
    __syncthreads();
    const int n = sh.n;
    // rank sort by (token, key) into scf/skey order: entry i goes to its rank
    __shared__ int rk_tok[kTreeMaxTerms];
    for (int i = threadIdx.x; i < n; i += kThreads) {
        int rank = 0;
        for (int j = 0; j < n; ++j)
            rank += sh.tok[j] < sh.tok[i] || (sh.tok[j] == sh.tok[i] && sh.skey[j] < sh.skey[i]);
        rk_tok[rank] = sh.tok[i];
        sh.scf[rank] = sh.cf[i];
    }
    __syncthreads();
    if (threadIdx.x == 0) {  // merge equal tokens, in order
        int m = 0;
        for (int i = 0; i < n; ++i) {
            if (m > 0 && sh.tok[m - 1] == rk_tok[i]) {
                sh.cf[m - 1] += sh.scf[i];
            } else {
                sh.tok[m] = rk_tok[i];
                sh.cf[m] = sh.scf[i];
                ++m;
            }
        }
        sh.nu = m;
    }
    __syncthreads();
    const int nu = sh.nu;
    // the first merged term at or after token v (binary search)
    auto first_at = [&](int64_t v) {
        int lo = 0, hi = nu;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((int64_t)sh.tok[mid] < v) lo = mid + 1; else hi = mid;
        }
        return lo;
    };
    const float gr = bad ? 0.f : ld_cg(P.tg + r);
    const RowRec rec = ld_cg(P.rows + r);
    const float gq = (nu == 0 && gr == 0.f) ? 0.f : gr * rec.izx;
    const float mx = rec.mx, c = P.ts.c;
    const bool dense = gq != 0.f && isfinite(mx);
    if constexpr (VEC) {
        const uint64_t pol = policy_evict_first();
        const int nvec = (int)(V / PV);
        for (int i = threadIdx.x; i < nvec; i += kThreads) {
            const int64_t v0 = (int64_t)i * PV;
            float o[PV];
            if (dense) {
                float f[PV];
                unpack<T>(ld_stream(x + v0, pol), f);
#pragma unroll
                for (int e = 0; e < PV; ++e) o[e] = gq * ex2((f[e] - mx) * c);
            } else {
#pragma unroll
                for (int e = 0; e < PV; ++e) o[e] = 0.f;
            }
            if (nu) {
                for (int k = first_at(v0); k < nu && sh.tok[k] < v0 + PV; ++k) {
#pragma unroll
                    for (int e = 0; e < PV; ++e)
                        if (v0 + e == sh.tok[k]) o[e] -= sh.cf[k];
                }
            }
            grad_store<T, G, PV>(g, v0, o, pol);
        }
    } else {
        for (int64_t v = threadIdx.x; v < V; v += kThreads) {
            float val = dense ? gq * ex2((elem_value(x, v) - mx) * c) : 0.f;
            if (nu) {
                const int k = first_at(v);
                if (k < nu && sh.tok[k] == v) val -= sh.cf[k];
            }
            if constexpr (sizeof(G) == 2)
                g[v] = __float2bfloat16_rn(val);
            else
                g[v] = val;
        }
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
};
inline size_t seq_smem_bytes(int N) { return (size_t)N * 32; }
__device__ __forceinline__ SeqKids seq_kids(unsigned char* base, int N) {
    SeqKids s;
    s.p = reinterpret_cast<double*>(base);
    s.q = s.p + N;
    s.A = reinterpret_cast<float2*>(s.q + N);
    s.tok = reinterpret_cast<int*>(s.A + N);
    s.kid = s.tok + N;
    return s;
}

__device__ __forceinline__ float2 two_floats(double a) {
    const float h = (float)a;
    return make_float2(h, (float)(a - (double)h));
}
// max(0, p - A q): the products are exact inside the multiply-adds, so A in
// two floats loses nothing of the double.
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
template <typename T, bool VEC>
__device__ void seq_stream(const Problem<T>& P, int r, Ring* rg, float4* tab, const SeqMass& sm) {
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
                        const SeqMass& sm, int lane) {
    const Located loc = table_locate(tab, P.nch, 0, 0.f, P.ts.c, S, u, lane);
    if (loc.ch < 0) return -1;
    return warp_rescan<T, VEC, true, true>(P.draft + (int64_t)r * P.V, P.target + (int64_t)r * P.V,
                                           P.V, loc.ch, loc.tc, sm, lane, policy_evict_normal());
}

// The decision at node u = row r (block, after the row's pass): tries its
// children in turn.  Per tried child tnode[].lq = alpha, .acc, .zp = 1 (0 for
// the others), for every child .la; tlist[r] = the accepted child, 0 if u has
// no children, -1 if all were rejected, with the correction token in
// es.corr[r].
template <typename T, bool VEC>
__device__ void tree_seq_row(const Problem<T>& P, int r, Ring* rg, float4* tab, SeqCtl& ct,
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
        s.tok[i] = tok;
        s.p[i] = p;
        s.q[i] = q;
        P.tnode[n] = nr;
    }
    __syncthreads();
    const MassRes mr{rec.mx, rec.my, rec.izx, rec.izy, c};
    for (int i = 0; i < m; ++i) {
        if (threadIdx.x == 0) {
            const int n = n0 + s.kid[i], t = s.tok[i];
            int before = -1;  // the earlier sibling that removed t, if any
            for (int j = 0; j < i && before < 0; ++j)
                if (s.tok[j] == t) before = j;
            const double Q = ct.Q, A = ct.A, Tm = ct.T;
            double alpha = 0.0;
            if (!rec.flags && t >= 0 && t < V) {
                const double At = before >= 0 ? (double)s.A[before].x + (double)s.A[before].y : A;
                const double pi = fmax(0.0, s.p[i] - At * s.q[i]) / Tm;
                const double qi = before >= 0 || !(Q > 0.0) ? 0.0 : s.q[i] / Q;
                alpha = qi > 0.0 ? fmin(1.0, pi / qi) : (pi > 0.0 ? 1.0 : 0.0);
            }
            const bool a = __ldg(P.u_accept + n) <= alpha && !rec.flags;
            P.tnode[n].lq = (float)alpha;
            P.tnode[n].acc = a ? 1 : 0;
            P.tnode[n].zp = 1;
            if (a) ct.next = s.kid[i];
            ct.An = A + (Q > 0.0 ? Tm / Q : 0.0);
            const float2 h = two_floats(ct.An);
            ct.ah = h.x;
            ct.al = h.y;
            if (before < 0) ct.Q = Q - s.q[i];
        }
        __syncthreads();
        if (ct.next > 0) break;
        if (!rec.flags) {
            // T_{i+1} (one read of the row); the draw after the last rejection
            const float uc = __ldg(P.u_correct + n0 + s.kid[i]);
            const SeqMass sm{mr, ct.ah, ct.al, s.tok, s.A, i};
            seq_stream<T, VEC>(P, r, rg, tab, sm);
            if (warp == 0) {
                const TableSum Rt = table_sum(tab, P.nch, 0, 0.f, c, lane);
                // (no mass left: p_i is kept, and the draw is from it)
                const int tok = i < m - 1 ? -1
                                : Rt.Z > 0.0 ? seq_draw<T, VEC>(P, r, tab, Rt, uc, sm, lane)
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
                        Pt.Z > 0.0 ? seq_draw<T, VEC>(P, r, tab, Pt, uc, keep, lane) : -1;
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

// One block per node row (a leaf's row only for the statistics output; the
// row the bonus token needs is then read by k_tree_seq).
// What bounds it: the row reads and row tails (3840 rows of 2 x 64 KB), and
// the reads after a rejection, which come from L2.  64 trees of 60 nodes,
// V = 32000: 0.244 ms a call; 5.46 ms with the rule run along the path by one
// block per tree, in an fp64 recursion per element over the earlier siblings.
template <typename T, bool VEC>
__global__ void __launch_bounds__(kThreads) k_tree_seq_rows(Problem<T> P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ RowShared sh;
    __shared__ SeqCtl ct;
    Ring* rg;
    float4* tab;
    smem_views<VEC>(dsm, rg, tab, P.timeout_ns);
    const SeqKids kids = seq_kids(reinterpret_cast<unsigned char*>(tab + P.nch), P.N);
    const int r = blockIdx.x, N = P.N, b = r / N, u = r - b * N;
    int need = P.tout.row_stats != nullptr;
    for (int n = u + 1 + threadIdx.x; n < N && !need; n += kThreads)
        need = __ldg(P.parent + (int64_t)b * N + n) == u;
    if (!__syncthreads_or(need)) {
        if (threadIdx.x == 0) P.tlist[r] = 0;
        return;
    }
    row_pass<T, VEC, true, kNoToken, false>(P, r, rg, tab, sh);
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
template <typename T, bool VEC>
__global__ void __launch_bounds__(kThreads) k_tree_seq(Problem<T> P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ RowShared rsh;
    Ring* rg;
    float4* tab;
    smem_views<VEC>(dsm, rg, tab, P.timeout_ns);
    TreeSeqShared& sh = *reinterpret_cast<TreeSeqShared*>(tab + P.nch);
    const int N = P.N, b = blockIdx.x, n0 = b * N;
    const vsd_tree_outputs& o = P.tout;
    if (!tree_load<T>(P, b, sh.t)) {
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
    if (leaf && !P.tout.row_stats) {  // the leaf's row, for the bonus token
        row_pass<T, VEC, true, kNoToken, false>(P, n0 + best, rg, tab, rsh);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        o.deepest[b] = best;
        o.accept_len[b] = sh.t.depth[best];
        const int tok = leaf ? ld_cg(P.rows + n0 + best).ps : P.es.corr[n0 + best];
        if (!leaf) o.corr_tokens[n0 + sh.lastkid] = tok;
        o.bonus[b] = tok;
    }
}

}  // namespace vsd
