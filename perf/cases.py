"""The calls whose speed matters here, as a user's program makes them.

Kinds of a case (its "kind"):
  em      the fused E-step + M-step (estep_mstep) on logits in device memory
  steps   the same work through the three separate calls (sample_paths,
          verify_paths, weighted_loss_fwd_bwd)
  tree    verification of draft trees (verify_tree), both sibling rules
  tree_em the E-step + M-step over draft trees (tree_estep_mstep)
  head    the LM head with the E-step + M-step (lmhead_estep_mstep), and with
          "train" its backward too (no dense gradient then)
  bwd     the LM head's backward alone (lmhead_backward), after an E-step +
          M-step on bf16 draft logits

listed() gives the sizes of the repository's workloads and a few between them,
draw(rng) more of the same ranges.  Inputs are the seeded recipes of
paper_2602_05774_gb300/inputs.py; plans, workspaces and output tensors are made
once per state, as a training or serving loop would hold them.

exact(case, seed) is the method in float64 with plain torch, and shares no code
with the library.  What depends on a draw that float32 cannot tell apart is
None there: at Zipf-shaped logits (a third of the mass on tokens narrower than
1e-6) and behind the LM head, whose bf16 logits round differently for another
order of summation.  And so are the weights, and the loss and gradient made with
them, where bf16 rows are compared with the greedy reference of the same rows:
there log kappas of different tokens are equal but for rounding (differences of
bf16 logits take few values), and either outcome of Algorithm 2's comparison is
right.
"""
import math

import torch

from paper_2602_05774_gb300 import inputs, vsd

DEV = "cuda"
W_BASE, TAU = 1.05, 0.2  # the defaults of vsd.params()


# ------------------------------------------------------------------ the cases
def _em(name, B, K, D, V, dtype="bf16", logits="spiked", T=1.0, kl=0.0, ref=False, kind="em"):
    c = dict(kind=kind, B=B, K=K, D=D, V=V, dtype=dtype, logits=logits, T=T, kl=kl, ref=ref)
    return dict(c, name=name) if name else c


def _tree(name, kind, B, N, depth, V, rule="independent", stats=False, T=1.0, dtype="bf16"):
    c = dict(kind=kind, B=B, N=N, depth=depth, topk=8, V=V, dtype=dtype, rule=rule, stats=stats,
             T=T)
    return dict(c, name=name) if name else c


def _head(name, kind, B, K, D, V, H, train=False, T=1.0):
    c = dict(kind=kind, B=B, K=K, D=D, V=V, H=H, train=train, T=T)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: 32 rows of 1024 float32 logits, latency throughout
        _em("em_tiny", 2, 4, 4, 1024, "f32", "gauss"),
        # a vocabulary that no 16-byte load divides, float32, an odd number of rows
        _em("em_ragged_f32", 5, 6, 7, 32003, "f32", "gauss", T=0.7),
        # a 32k vocabulary, an ordinary training step of 768 rows
        _em("em_vocab32k", 16, 8, 6, 32000),
        # the same with VSD (KL)'s top-10 term and Algorithm 2's reference from its own rows
        _em("em_kl_ref", 16, 8, 6, 32000, kl=0.1, ref=True),
        # a 128k vocabulary, Zipf-shaped, 4096 rows: the headline workload
        _em("em_vocab128k", 32, 16, 8, 128256, logits="zipf", T=0.7),
        # sampling, verification and loss by separate calls, as a program that
        # inspects or replaces one of the steps makes them
        _em("steps_vocab32k", 16, 8, 6, 32000, kind="steps"),
        # serving: 64 trees of 60 nodes, branch by branch
        _tree("tree60", "tree", 64, 60, 7, 32000),
        # serving without loss: the sequential sibling rule on the same trees
        _tree("tree60_seq", "tree", 64, 60, 7, 32000, rule="sequential", stats=True),
        # training on trees, every node a proposal
        _tree("tree60_em", "tree_em", 64, 60, 7, 32000),
        # the draft head's forward with the E-step + M-step and a dense gradient
        _head("head_em", "head", 64, 8, 8, 32000, 4096),
        # the draft head's whole training step: forward, E-step + M-step, backward
        _head("head_train", "head", 64, 8, 8, 32000, 4096, train=True),
        # the backward of a smaller step whose sizes no tile divides
        _head("bwd_ragged", "bwd", 12, 8, 7, 32000, 2888),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["em", "em", "em", "steps", "tree", "tree_em", "head", "bwd"])
    T = rng.choice([1.0, 1.0, 0.7, round(rng.uniform(0.3, 1.5), 2)])
    if kind in ("em", "steps"):
        V = _log_int(rng, 1000, 128256)
        V = rng.choice([V, V // 8 * 8, V // 8 * 8])
        K, D = rng.randint(2, 16), rng.randint(2, 10)
        dtype = rng.choice(["bf16", "bf16", "f32"])
        B = _log_int(rng, 1, max(1, min(64, (250_000_000 if dtype == "f32" else 500_000_000)
                                        // (K * D * V))))
        logits = rng.choice(["gauss", "spiked", "zipf"])
        if kind == "steps":
            return _em(None, B, K, D, V, dtype, logits, T, kind="steps")
        return _em(None, B, K, D, V, dtype, logits, rng.choice([T, T, T, 0.0]),
                   kl=rng.choice([0.0, 0.0, 0.1]), ref=rng.random() < 0.25)
    if kind in ("tree", "tree_em"):
        V = _log_int(rng, 4000, 64000)
        V = rng.choice([V, V // 8 * 8, V // 8 * 8])
        N, depth = rng.randint(10, 64), rng.randint(3, 8)
        rule = rng.choice(["independent", "sequential"]) if kind == "tree" else "independent"
        return _tree(None, kind, _log_int(rng, 1, max(1, min(64, 120_000_000 // (N * V)))), N,
                     depth, V, rule, rng.random() < 0.5 and kind == "tree", T,
                     rng.choice(["bf16", "bf16", "f32"]))
    V, H = _log_int(rng, 4000, 32000) // 8 * 8, _log_int(rng, 512, 4096) // 8 * 8
    K, D = rng.randint(2, 8), rng.randint(2, 8)
    B = _log_int(rng, 1, 64)
    return _head(None, kind, B, K, D, V, H, train=kind == "head" and rng.random() < 0.5, T=T)


# ------------------------------------------------------------------ inputs
def _problem(case, seed):
    """The inputs of a case, from the seed alone."""
    k = case["kind"]
    if k in ("em", "steps"):
        return inputs.linear_problem(case["B"], case["K"], case["D"], case["V"], case["dtype"],
                                     case["logits"], DEV, seed)
    if k in ("tree", "tree_em"):
        return inputs.tree_problem(case["B"], case["N"], case["depth"], case["topk"], case["V"],
                                   DEV, seed, case["dtype"])
    p = inputs.lmhead_problem(case["B"], case["K"], case["D"], case["V"], case["H"], DEV, seed)
    if k == "bwd":  # the draft logits of that backward: the spiked recipe
        d = inputs.linear_problem(case["B"], case["K"], case["D"], case["V"], "bf16", "spiked",
                                  DEV, seed)
        p.update({n: d[n] for n in ("draft", "target", "u_draft", "u_accept", "u_correct")})
        # a reference of the caller's own (Algorithm 2): log kappas that fall with the length
        u = inputs.uniforms(case["B"] * case["D"], DEV, seed + 6).view(case["B"], case["D"])
        p["ref"] = -u.cumsum(1).contiguous()
    return p


def _ref_problem(case, seed):
    """The rows along the greedy reference path, one of D rows per prefix."""
    return inputs.linear_problem(case["B"], 1, case["D"], case["V"], case["dtype"],
                                 case["logits"], DEV, seed + 1000)


def prepare(case, seed):
    s = dict(case=case, p=_problem(case, seed))
    p, k, V = s["p"], case["kind"], case["V"]
    if k in ("tree", "tree_em"):
        lay = vsd.layout(case["B"], V=V, N=case["N"], parent=p["parent"])
        s["ws"] = vsd.new_workspace(lay, torch.device(DEV))
        if k == "tree":
            s["out"] = vsd.tree_outputs(case["B"], case["N"], DEV, row_stats=case["stats"])
        else:
            s["prm"] = vsd.params(like=p["draft"])
        return s
    B, K, D = case["B"], case["K"], case["D"]
    s["ws"] = vsd.new_workspace(vsd.layout(B, K, D, V), torch.device(DEV))
    like = p["target"]
    s["prm"] = vsd.params(like=like, kl_weight=case.get("kl", 0.0))
    if k == "em":
        s["out"] = vsd.linear_outputs(B, K, D, V, DEV, grad_dtype=like.dtype,
                                      kl=case["kl"] != 0)
        if case["ref"]:
            s["ref"] = _ref_problem(case, seed)
            s["ref_ws"] = vsd.new_workspace(vsd.layout(B, 1, D, V), torch.device(DEV))
    elif k == "head":
        R, H = B * K * D, case["H"]
        s["out"] = vsd.linear_outputs(B, K, D, V, DEV, grad=not case["train"])
        s["logits"] = torch.empty(R, V, dtype=torch.bfloat16, device=DEV)
        if case["train"]:
            s["dh"] = torch.empty(R, H, device=DEV)
            s["dw"] = torch.empty(V, H, device=DEV)
    elif k == "bwd":
        R, H = B * K * D, case["H"]
        s["dh"], s["dw"] = torch.empty(R, H, device=DEV), torch.empty(V, H, device=DEV)
        vsd.estep_mstep(p["draft"], p["target"], p["u_draft"], p["u_accept"], p["u_correct"], K,
                        D, case["T"], ref_logkappa=p["ref"], prm=s["prm"], workspace=s["ws"],
                        grad=False)
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case, p = s["case"], s["p"]
    k, T = case["kind"], case["T"]
    if k == "tree":
        rule = vsd.TREE_SEQUENTIAL if case["rule"] == "sequential" else vsd.TREE_INDEPENDENT
        return vsd.verify_tree(p["draft"], p["target"], p["parent"], p["tokens"], p["u_accept"],
                               p["u_correct"], T, workspace=s["ws"], out=s["out"], rule=rule)
    if k == "tree_em":
        return vsd.tree_estep_mstep(p["draft"], p["target"], p["parent"], p["tokens"],
                                    p["u_accept"], p["u_correct"], T, prm=s["prm"],
                                    workspace=s["ws"])
    K, D = case["K"], case["D"]
    if k == "em":
        ref = None
        if case["ref"]:
            ref = vsd.reference_logkappa(s["ref"]["draft"], s["ref"]["target"], case["B"], D, T,
                                         workspace=s["ref_ws"])
        return vsd.estep_mstep(p["draft"], p["target"], p["u_draft"], p["u_accept"],
                               p["u_correct"], K, D, T, ref_logkappa=ref, prm=s["prm"],
                               workspace=s["ws"], out=s["out"])
    if k == "steps":
        a = vsd.sample_paths(p["draft"], p["u_draft"], K, D, T, workspace=s["ws"])
        o = vsd.verify_paths(p["draft"], p["target"], a["tokens"], p["u_accept"], p["u_correct"],
                             K, D, T, workspace=s["ws"])
        m = vsd.weighted_loss_fwd_bwd(p["draft"], o, K, D, T, prm=s["prm"], workspace=s["ws"])
        return dict(o, sampled=a, **m)
    if k == "head":
        o = vsd.lmhead_estep_mstep(p["hidden"], p["weight"], p["target"], p["u_draft"],
                                   p["u_accept"], p["u_correct"], K, D, T, prm=s["prm"],
                                   workspace=s["ws"], out=s["out"], draft_logits=s["logits"])
        if case["train"]:
            o = dict(o, **vsd.lmhead_backward(p["hidden"], p["weight"], s["logits"], K, D, T,
                                              s["ws"], prm=s["prm"], d_hidden=s["dh"],
                                              d_weight=s["dw"]))
        return o
    return vsd.lmhead_backward(p["hidden"], p["weight"], p["draft"], K, D, T, s["ws"],
                               prm=s["prm"], d_hidden=s["dh"], d_weight=s["dw"])


# ------------------------------------------------------------------ work
def work(case):
    """Each input read once, each output written once (per-row scalars are a
    few tens of bytes a row and are counted as 64)."""
    k, V = case["kind"], case["V"]
    e = 4 if case.get("dtype") == "f32" else 2
    if k in ("tree", "tree_em"):
        R = case["B"] * case["N"]
        # rows with children are what a tree verification cannot do without:
        # about half of the nodes; every row with statistics or a gradient
        rows = R if case["stats"] or k == "tree_em" else R // 2
        g = R * V * e if k == "tree_em" else 0
        return dict(bytes=2 * rows * V * e + g + 64 * R, flops=0)
    R = case["B"] * case["K"] * case["D"]
    if k in ("em", "steps"):
        ref = 2 * case["B"] * case["D"] * V * e if case["ref"] else 0
        return dict(bytes=3 * R * V * e + ref + 64 * R, flops=0)
    H = case["H"]
    mm = 2 * R * V * H
    if k == "bwd":
        return dict(bytes=2 * (R * V + R * H + V * H) + 4 * (R * H + V * H), flops=2 * mm)
    fwd = 2 * (R * H + V * H + 2 * R * V) + 64 * R
    if not case["train"]:
        return dict(bytes=fwd + 2 * R * V, flops=mm)
    return dict(bytes=fwd + 4 * (R * H + V * H), flops=3 * mm)


def tolerance(case):
    """About four times what run() shows against exact()."""
    if case["kind"] in ("head", "bwd") or (case["kind"] != "tree" and case["dtype"] == "bf16"):
        # bf16 logits or gradients, rounded once: half an ulp, 2^-9, in the
        # worst element and 1.7e-3 in the mean
        return dict(rel=7e-3, max=2e-2, differ=2e-3)
    # float32 throughout: up to 5e-7 seen (log kappas, whose terms cancel)
    return dict(rel=2e-6, max=1e-4, differ=2e-3)


# ------------------------------------------------------------------ float64
def _log_softmax(x, T):
    return torch.log_softmax(x.double() / T, dim=-1)


def _pick(prob, u):
    """Smallest v with u < F(v), per row."""
    F = prob.cumsum(-1)
    i = torch.searchsorted(F, u.double().view(-1, 1), right=True).view(-1)
    return i.clamp(max=prob.shape[-1] - 1)


def _residual(p, q):
    r = (p - q).clamp(min=0)
    m = r.sum(-1, keepdim=True)
    return torch.where(m > 0, r / m, p)


def _at(x, i):
    return x.gather(-1, i.view(-1, 1)).view(-1)


def _stats(d, t, T):
    a, b = d.double(), t.double()
    ma, mb = a.amax(-1), b.amax(-1)
    return torch.stack([ma, torch.logsumexp((a - ma[:, None]) / T, -1), mb,
                        torch.logsumexp((b - mb[:, None]) / T, -1)], 1)


def _log_ratio(lp, lq, tok, greedy, top_p=None, top_q=None):
    """log min(1, p/q) at tok; at T = 0 of the one-hot limits."""
    if greedy:
        p, q = (tok == top_p).double(), (tok == top_q).double()
        return torch.where(q > 0, p / q, torch.where(p > 0, 1.0, math.nan)).log().clamp(max=0)
    return (_at(lp, tok) - _at(lq, tok)).clamp(max=0)


def _zeta(lqp, dim):
    return torch.softmax(lqp.exp() / TAU, dim)


def _beta(ot, op, dim):
    num = (op * ot).sum(dim, keepdim=True) - op * ot
    den = op.sum(dim, keepdim=True) - op
    # exact zeros: no other valid proposal
    some = ((op > 0).sum(dim, keepdim=True) - (op > 0).long()) > 0
    return torch.where(some, num / torch.where(some, den, 1.0), 0.0)


def _exact_linear(draft, target, u_draft, u_accept, u_correct, B, K, D, T, ref=None, kl=0.0,
                  topk=10):
    greedy, Tq = T == 0.0, T if T > 0 else 1.0
    lq, lp = _log_softmax(draft, Tq), _log_softmax(target, Tq)
    vb, va = target.float().argmax(-1), draft.float().argmax(-1)
    # argmax: the lowest index among equals
    vb = (target == target.gather(-1, vb[:, None])).int().argmax(-1)
    va = (draft == draft.gather(-1, va[:, None])).int().argmax(-1)
    tok = va if greedy else _pick(lq.exp(), u_draft)
    la = _log_ratio(lp, lq, tok, greedy, vb, va)
    acc = u_accept.double() <= la.exp()
    A = acc.view(B * K, D).long().cumprod(1).sum(1)
    d = torch.arange(D, device=tok.device).repeat(B * K)
    An = A.repeat_interleave(D)
    if greedy:
        other = vb
    else:
        other = _pick(lp.exp(), u_correct)
        at = ((d == An).nonzero()).view(-1)
        if at.numel():
            other[at] = _pick(_residual(lp[at].exp(), lq[at].exp()), u_correct[at])
    corr = torch.where(d < An, tok, other)
    lc = _log_ratio(lp, lq, corr, greedy, vb, va)
    lr = _log_ratio(lp, lq, vb, greedy, vb, va)
    run_ = lambda x: x.view(B, K, D).cumsum(-1)  # noqa: E731
    lk, lkc, lkr = run_(la), run_(lc), run_(lr)
    if ref is not None:
        lkr = ref.double().view(B, 1, D).expand(B, K, D)
    qt, qc = _at(lq, tok), _at(lq, corr)
    lqt, lqc = run_(qt), run_(qc)
    w = W_BASE ** torch.arange(1, D + 1, device=tok.device, dtype=torch.float64)
    ot = (lk >= lkr).double()
    op = torch.where(ot > 0, w.expand(B, K, D), (lkc >= lkr).double() * w)
    beta, zeta = _beta(ot, op, 1), _zeta(lqt, 1)
    N = op.sum((1, 2))
    J = (op * (torch.where(ot > 0, lqt, torch.where(op > 0, lqc, 0.0)) - beta * zeta * lqt)).sum(
        (1, 2))
    loss = torch.where(N > 0, -J / torch.where(N > 0, N, 1.0), 0.0)
    s = torch.where(N > 0, 1.0 / torch.where(N > 0, N, 1.0), 0.0).view(B, 1, 1) / B
    tail = lambda x: x.flip(-1).cumsum(-1).flip(-1).reshape(-1)  # noqa: E731
    pt, pc, ng = tail(-op * ot * s), tail(-op * (1 - ot) * s), tail(op * beta * zeta * s)
    g = lq.exp_().mul_(-(pt + pc + ng)[:, None])  # lq is not needed any more
    g.scatter_add_(1, tok[:, None], (pt + ng)[:, None])
    g.scatter_add_(1, corr[:, None], pc[:, None])
    g /= Tq
    out = dict(tokens=tok, logq_tok=qt, alpha=la.exp(), accept=acc.long(), accept_len=A,
               corr_tokens=corr, logq_corr=qc, alpha_corr=lc.exp(), logkappa=lk.reshape(-1),
               logkappa_corr=lkc.reshape(-1), logkappa_ref=lkr.reshape(-1), ref_tokens=vb,
               expected_len=lk.exp().sum(-1).view(-1), row_stats=_stats(draft, target, Tq),
               weights=torch.stack([ot, op, beta, zeta], -1).transpose(1, 2).contiguous(),
               grad=g)
    if kl:
        val, top = target.float().sort(dim=-1, descending=True, stable=True)
        top, val = top[:, :topk], val[:, :topk].double()
        ph = torch.softmax(val / Tq, -1)
        lqh = torch.log_softmax(draft.double().gather(1, top) / Tq, -1)
        row = -(ph * lqh).sum(-1)
        g.scatter_add_(1, top, (lqh.exp() - ph) * (kl / (B * K * Tq)))
        loss = loss + kl * row.view(B, -1).sum(1) / K
        out["kl_loss"] = row
    out["loss"] = torch.cat([loss, loss.mean().view(1)])
    return out


def _exact_reference(p, B, D, T):
    Tq = T if T > 0 else 1.0
    lq, lp = _log_softmax(p["draft"], Tq), _log_softmax(p["target"], Tq)
    top = p["target"].float().argmax(-1)
    top = (p["target"] == p["target"].gather(-1, top[:, None])).int().argmax(-1)
    if T == 0:
        return torch.zeros(B, D, dtype=torch.float64, device=top.device)
    return _log_ratio(lp, lq, top, False).view(B, D).cumsum(1)


def _depths(parent):
    dep = torch.zeros_like(parent)
    for n in range(1, parent.shape[1]):
        dep[:, n] = dep.gather(1, parent[:, n:n + 1]).view(-1) + 1
    return dep


def _bonus(p, T, dep, pa, corr, which):
    """Deepest accepted node (lowest index), its depth and the token after it;
    `which` picks the child whose correction that is: the first or the last."""
    B, N = dep.shape
    par = p["parent"].long()
    deep = torch.where(pa, dep, -1).argmax(1)
    best = torch.where(pa, dep, -1).max(1).values
    # the lowest index among equals
    deep = (torch.where(pa, dep, -1) == best[:, None]).int().argmax(1)
    rows = torch.arange(B, device=dep.device) * N + deep
    leaf = _pick(_log_softmax(p["target"][rows], T).exp(), p["u_correct"].view(-1)[rows])
    kids = par == deep[:, None]
    kid = kids.int().argmax(1) if which == "first" else N - 1 - kids.flip(1).int().argmax(1)
    at_kid = corr.gather(1, kid[:, None]).view(-1)
    return deep, best, torch.where(kids.any(1) & (at_kid >= 0), at_kid, leaf)


def _exact_tree(case, p):
    B, N, T = case["B"], case["N"], case["T"]
    par, tok = p["parent"].long(), p["tokens"].long()
    base = torch.arange(B, device=par.device) * N
    lq, lp = _log_softmax(p["draft"], T), _log_softmax(p["target"], T)
    dep = _depths(par)
    rows = (base[:, None] + par.clamp(min=0)).view(-1)
    la = (lp[rows, tok.view(-1)] - lq[rows, tok.view(-1)]).clamp(max=0).view(B, N)
    la[:, 0] = 0
    lk = la.clone()
    for n in range(1, N):
        lk[:, n] += lk.gather(1, par[:, n:n + 1]).view(-1)
    corr = torch.full_like(tok, -1)
    pa = torch.zeros(B, N, dtype=torch.bool, device=par.device)
    pa[:, 0] = True
    if case["rule"] == "independent":
        alpha, acc = la.exp(), p["u_accept"].double() <= la.exp()
        acc[:, 0] = True
        for n in range(1, N):
            up = pa.gather(1, par[:, n:n + 1]).view(-1)
            pa[:, n] = up & acc[:, n]
            b = (up & ~acc[:, n]).nonzero().view(-1)
            if b.numel():
                r = base[b] + par[b, n]
                corr[b, n] = _pick(_residual(lp[r].exp(), lq[r].exp()), p["u_correct"][b, n])
        deep, best, bonus = _bonus(p, T, dep, pa, corr, "first")
    else:
        alpha = torch.zeros(B, N, dtype=torch.float64, device=par.device)
        alpha[:, 0] = 1
        acc = pa.clone()
        pl, ua = par.tolist(), p["u_accept"].double().tolist()
        tl = tok.tolist()
        for b in range(B):
            u = 0
            while u is not None:
                kids = [n for n in range(u + 1, N) if pl[b][n] == u]
                r, nxt = b * N + u, None
                q, pp = lq[r].exp(), lp[r].exp()
                for n in kids:
                    t = tl[b][n]
                    pt, qt = float(pp[t]), float(q[t])
                    a = min(1.0, pt / qt) if qt > 0 else float(pt > 0)
                    alpha[b, n] = a
                    if ua[b][n] <= a:
                        acc[b, n] = pa[b, n] = True
                        nxt = n
                        break
                    pp = _residual(pp[None], q[None])[0]
                    q[t] = 0
                    q = q / q.sum()
                if kids and nxt is None:
                    n = kids[-1]
                    corr[b, n] = _pick(pp[None], p["u_correct"][b, n:n + 1])[0]
                u = nxt
        deep, best, bonus = _bonus(p, T, dep, pa, corr, "last")
    out = dict(alpha=alpha, accept=acc.long(), path_accept=pa.long(), logkappa=lk,
               corr_tokens=corr, deepest=deep, accept_len=best, bonus=bonus)
    if case["stats"]:
        out["row_stats"] = _stats(p["draft"], p["target"], T)
    return out


def _exact_tree_em(case, p):
    B, N, T, V = case["B"], case["N"], case["T"], case["V"]
    par, tok = p["parent"].long(), p["tokens"].long()
    dev = par.device
    base = torch.arange(B, device=dev) * N
    lq, lp = _log_softmax(p["draft"], T), _log_softmax(p["target"], T)
    dep = _depths(par)
    top = p["target"].float().argmax(-1)
    top = (p["target"] == p["target"].gather(-1, top[:, None])).int().argmax(-1)
    z = lambda: torch.zeros(B, N, dtype=torch.float64, device=dev)  # noqa: E731
    qt, qc, lk, lkc, lkr, pq, pc = z(), z(), z(), z(), z(), z(), z()
    corr = torch.full_like(tok, -1)
    pa = torch.zeros(B, N, dtype=torch.bool, device=dev)
    pa[:, 0] = True
    for n in range(1, N):
        a = par[:, n]
        up = lambda x: x.gather(1, a[:, None]).view(-1)  # noqa: E731
        r = base + a
        t = tok[:, n]
        la = (lp[r, t] - lq[r, t]).clamp(max=0)
        ok = p["u_accept"][:, n].double() <= la.exp()
        pa[:, n] = ok & up(pa)
        pr, qr = lp[r].exp(), lq[r].exp()
        first = up(pa) & ~ok
        c = _pick(torch.where(first[:, None], _residual(pr, qr), pr), p["u_correct"][:, n])
        c = torch.where(pa[:, n], t, c)
        corr[:, n] = c
        qt[:, n], qc[:, n] = lq[r, t], lq[r, c]
        lk[:, n] = up(lk) + la
        lkc[:, n] = up(lkc) + (lp[r, c] - lq[r, c]).clamp(max=0)
        lkr[:, n] = up(lkr) + (lp[r, top[r]] - lq[r, top[r]]).clamp(max=0)
        pq[:, n], pc[:, n] = up(pq) + qt[:, n], up(pc) + qc[:, n]
    w = W_BASE ** dep.double()
    real = dep > 0
    ot = ((lk >= lkr) & real).double()
    op = torch.where(ot > 0, w, ((lkc >= lkr) & real).double() * w)
    beta, zeta = z(), z()
    for l in range(1, int(dep.max()) + 1):
        m = dep == l
        o, t = torch.where(m, op, 0.0), torch.where(m, ot, 0.0)
        beta = torch.where(m, _beta(t, o, 1), beta)
        zz = torch.softmax(torch.where(m, pq.exp() / TAU, -math.inf), 1)
        zeta = torch.where(m, zz, zeta)
    Nb = op.sum(1)
    J = (op * (torch.where(ot > 0, pq, pc) - beta * zeta * pq)).sum(1)
    some = Nb > 0
    loss = torch.where(some, -J / torch.where(some, Nb, 1.0), 0.0)
    s = torch.where(some, 1.0 / torch.where(some, Nb, 1.0), 0.0)[:, None] / B
    st, sc, sn = -op * ot * s, -op * (1 - ot) * s, op * beta * zeta * s
    for x in (st, sc, sn):  # over each node's subtree
        for n in range(N - 1, 0, -1):
            x.scatter_add_(1, par[:, n:n + 1], x[:, n:n + 1])
    g = torch.zeros(B * N, V, dtype=torch.float64, device=dev)
    tot = z()
    for n in range(1, N):
        r = base + par[:, n]
        g[r, tok[:, n]] += st[:, n] + sn[:, n]
        g[r, corr[:, n]] += sc[:, n]
        tot.view(-1)[r] += st[:, n] + sc[:, n] + sn[:, n]
    g -= tot.view(-1, 1) * lq.exp_()
    g /= T
    W = torch.stack([ot, op, beta, zeta], -1)
    return dict(corr_tokens=corr, logq_tok=qt, logq_corr=qc, logkappa=lk, logkappa_corr=lkc,
                logkappa_ref=lkr, weights=W, loss=torch.cat([loss, loss.mean().view(1)]), grad=g)


ROW_ONLY = ("row_stats", "ref_tokens", "logkappa_ref")  # what no draw decides
MADE_OF_TIES = ("weights", "loss", "grad")  # bf16 rows against their own reference


def exact(case, seed):
    k, T = case["kind"], case["T"]
    p = _problem(case, seed)
    if k == "tree":
        return _exact_tree(case, p)
    if k == "tree_em":
        o = _exact_tree_em(case, p)
        if case["dtype"] == "bf16":
            o.update((n, None) for n in MADE_OF_TIES)
        return o
    B, K, D = case["B"], case["K"], case["D"]
    if k == "head":
        x = p["hidden"].double() @ p["weight"].double().t()
        R, V, H = x.shape[0], case["V"], case["H"]
        lq, lp = _log_softmax(x, T), _log_softmax(p["target"], T)
        top = p["target"].float().argmax(-1)
        top = (p["target"] == p["target"].gather(-1, top[:, None])).int().argmax(-1)
        lkr = _log_ratio(lp, lq, top, False).view(B, K, D).cumsum(-1)
        names = ["tokens", "accept_len", "corr_tokens", "logkappa", "loss", "logq_tok", "alpha",
                 "accept", "logq_corr", "alpha_corr", "logkappa_corr", "expected_len", "weights"]
        names += ["d_hidden", "d_weight"] if case["train"] else ["grad"]
        # the statistics are those of the logits as rounded to bf16
        o = dict(draft_logits=x, row_stats=_stats(x.bfloat16(), p["target"], T),
                 ref_tokens=top, logkappa_ref=lkr.reshape(-1))
        return dict(o, **{n: None for n in names})
    ref = None
    if k == "em" and case["ref"]:
        ref = _exact_reference(_ref_problem(case, seed), B, D, T)
    elif k == "bwd":
        ref = p["ref"]
    o = _exact_linear(p["draft"], p["target"], p["u_draft"], p["u_accept"], p["u_correct"], B, K,
                      D, T, ref, case.get("kl", 0.0))
    if k == "bwd":
        g = o["grad"]
        return dict(d_hidden=g @ p["weight"].double(), d_weight=g.t() @ p["hidden"].double())
    if case["logits"] == "zipf":
        o = {n: (v if n in ROW_ONLY else None) for n, v in o.items()}
    elif case["dtype"] == "bf16" and ref is None:
        o.update((n, None) for n in MADE_OF_TIES)
    if k == "steps":
        st = o["row_stats"].clone()
        st[:, 2:] = 0
        o["sampled"] = dict(tokens=o["tokens"], logq_tok=o["logq_tok"], row_stats=st)
    return o
