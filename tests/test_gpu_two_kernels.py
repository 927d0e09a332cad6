"""The E-step + M-step as two kernels (short rows, small batches, no gradient)
and as the persistent kernel (long rows with a gradient): against the oracle at
the edges of the first, and against each other bit for bit."""
import numpy as np
import pytest
import torch

from tests.parity import compare_linear, mstep_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vsd():
    from paper_2602_05774_gb300 import build, vsd as v
    build.build_library()
    v.load()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    return v


def _call(vsd, p, T, prm, **kw):
    return vsd.estep_mstep(p["draft"], p["target"], p["u_draft"], p["u_accept"], p["u_correct"],
                           p["K"], p["D"], T, prm=prm, **kw)


@pytest.mark.parametrize("B,K,D,V,dtype,grad,kl", [
    (1, 1, 1, 65544, "bf16", "bf16", 0.0),   # one row in many gradient segments, ragged last chunk
    (1, 2, 1, 65537, "f32", "f32", 0.5),     # the same, rows not 16-byte aligned
    (2, 256, 1, 40, "f32", "bf16", 0.0),     # the most proposals
    (1, 5, 64, 24, "f32", "f32", 0.0),       # the deepest paths
    (2, 30, 17, 264, "bf16", "f32", 0.5),    # an M-step of several tiles
    (3, 3, 5, 8200, "bf16", "bf16", 0.5),    # top-K terms across gradient segments
])
def test_two_kernels_match_oracle(vsd, oracle, B, K, D, V, dtype, grad, kl):
    from paper_2602_05774_gb300 import inputs
    prob = inputs.linear_problem(B, K, D, V, dtype, "gauss", seed=V + K)
    f = lambda t: t.float().numpy()  # noqa: E731
    orc = oracle.linear(f(prob["draft"]), f(prob["target"]), 1.0, f(prob["u_draft"]),
                        f(prob["u_accept"]), f(prob["u_correct"]), K, D, kl_weight=kl, kl_topk=10)
    p = {k: (v.cuda() if torch.is_tensor(v) else v) for k, v in prob.items()}
    prm = vsd.params(grad_dtype=torch.float32 if grad == "f32" else torch.bfloat16, kl_weight=kl)
    ws = vsd.new_workspace(vsd.layout(B, K, D, V), "cuda")
    got = _call(vsd, p, 1.0, prm, workspace=ws)
    torch.cuda.synchronize()
    assert vsd.device_status(ws) == (0, 0)
    compare_linear(got, orc, B, K, D, V, 1.0, grad_dtype=grad, kl=kl != 0,
                   mstep_inputs=mstep_inputs(prob, kl_weight=kl, kl_topk=10) if kl
                   else mstep_inputs(prob))


@pytest.mark.parametrize("V,R,dtype,kind,kl,T", [
    (70000, 2048, "bf16", "spiked", 0.0, 1.0),
    (140000, 1024, "bf16", "zipf", 0.3, 0.7),   # two row segments
    (70001, 1024, "f32", "gauss", 0.3, 1.0),    # rows not 16-byte aligned (two kernels)
    (70000, 2048, "bf16", "spiked", 0.3, 0.0),  # greedy
])
def test_persistent_kernel_equals_two_kernels(vsd, V, R, dtype, kind, kl, T):
    """An aligned batch above the dispatch's size runs on the persistent kernel,
    each half of it on the two kernels: every result equal bit for bit (halving
    the batch doubles the gradient, an exact factor)."""
    from paper_2602_05774_gb300 import inputs
    K, D = 8, 8
    B = R // (K * D)
    p = inputs.linear_problem(B, K, D, V, dtype, kind, "cuda", seed=V)
    prm = vsd.params(like=p["draft"], kl_weight=kl)
    whole = _call(vsd, p, T, prm)
    none = _call(vsd, p, T, prm, grad=False)
    for n in none:
        if n != "grad":
            assert torch.equal(whole[n], none[n]), n
    h = R // 2
    for i in range(2):
        q = dict(p, **{k: p[k][i * h:(i + 1) * h] for k in
                       ("draft", "target", "u_draft", "u_accept", "u_correct")})
        part = _call(vsd, q, T, prm)
        assert torch.equal(whole["loss"][i * B // 2:(i + 1) * B // 2], part["loss"][:-1])
        a, b = whole["grad"][i * h:(i + 1) * h], part["grad"]
        assert torch.equal(2 * a, b)
        for n in ("tokens", "corr_tokens", "logkappa", "weights", "row_stats"):
            m = whole[n].view(2, -1)[i]
            assert torch.equal(m, part[n].reshape(-1)), n


@pytest.mark.parametrize("offset", ["target", "grad"])
def test_lmhead_with_unaligned_rows_waits_for_its_logits(vsd, offset):
    """Rows that start off a 16-byte boundary, behind the LM head: the row kernel
    starts before the head's product has ended and must not read the logits
    until then.  Equal bit for bit to the E-step + M-step on the logits left."""
    B, K, D, V, H = 32, 8, 8, 32000, 1024
    R = B * K * D
    g = torch.Generator(device="cuda").manual_seed(3)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    hidden = rnd(R, H).bfloat16()
    weight = (rnd(V, H) / H ** 0.5).bfloat16()
    off = lambda want: 1 if offset == want else 0  # noqa: E731
    target = torch.empty(R * V + 1, dtype=torch.bfloat16, device="cuda")
    target = target[off("target"):][:R * V].view(R, V).copy_(2 * rnd(R, V))
    u = [torch.rand(R, device="cuda", generator=g) for _ in range(3)]
    prm = vsd.params(like=target)
    for _ in range(3):
        logits = torch.full((R, V), float("nan"), dtype=torch.bfloat16, device="cuda")
        res = []
        for head in (True, False):
            ws = vsd.new_workspace(vsd.layout(B, K, D, V), "cuda")
            out = vsd.linear_outputs(B, K, D, V, "cuda", grad=False)
            buf = torch.empty(R * V + 1, dtype=torch.bfloat16, device="cuda")
            out["grad"] = buf[off("grad"):][:R * V].view(R, V)
            if head:
                vsd.lmhead_estep_mstep(hidden, weight, target, *u, K, D, 1.0, prm=prm,
                                       workspace=ws, out=out, draft_logits=logits)
            else:
                vsd.estep_mstep(logits, target, *u, K, D, 1.0, prm=prm, workspace=ws, out=out)
            torch.cuda.synchronize()
            assert vsd.device_status(ws) == (0, 0)
            res.append(out)
        for k, want in res[1].items():
            assert torch.equal(res[0][k], want), k


def test_mstep_scratch_is_its_own(vsd):
    """The M-step's scratch shares shared memory with the row stream's copies, but
    not with their barriers, and runs where the LM head's blocks have just left:
    every call gives all of the outputs that the E-step + M-step gives on the
    logits left behind.  (The head's own chunk statistics add the same terms in
    another order: running masses differ by up to 2^-23 on either side of boundaries
    that lie 1/V apart, so up to V 2^-22 of the draws, 0.8 %, may go the other way;
    the weights and log kappas of prefixes whose tokens agree lie within float32's
    sums of K D = 64 terms.)  With the barriers' words in the scratch, about one call in
    14 had a prefix whose zeta held them."""
    B, K, D, V, H = 64, 8, 8, 32000, 4096
    R = B * K * D
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g).bfloat16()  # noqa: E731
    hidden, weight, target = rnd(R, H), rnd(V, H) / 64, rnd(R, V) * 2
    u = [torch.rand(R, device="cuda", generator=g) for _ in range(3)]
    prm = vsd.params(like=target)
    ws = vsd.new_workspace(vsd.layout(B, K, D, V), "cuda")
    logits = torch.empty(R, V, dtype=torch.bfloat16, device="cuda")
    outs = [vsd.linear_outputs(B, K, D, V, "cuda", grad=False) for _ in range(60)]
    for o in outs:
        vsd.lmhead_estep_mstep(hidden, weight, target, *u, K, D, 1.0, prm=prm, workspace=ws,
                               out=o, draft_logits=logits)
    want = vsd.estep_mstep(logits, target, *u, K, D, 1.0, prm=prm, grad=False)
    torch.cuda.synchronize()
    assert vsd.device_status(ws) == (0, 0)
    first = outs[0]
    for o in outs[1:]:
        for k in want:
            assert torch.equal(o[k], first[k]), k
    same = torch.ones(B, dtype=torch.bool, device="cuda")
    for k in ("tokens", "accept", "corr_tokens", "ref_tokens"):
        differ = (first[k] != want[k]).view(B, K * D)
        assert differ.float().mean() < V * 2.0 ** -22, k
        same &= ~differ.any(dim=1)
    # (nor where Algorithm 2 compares log kappas that are equal but for rounding)
    same &= (first["weights"][..., :2] == want["weights"][..., :2]).view(B, -1).all(dim=1)
    assert same.float().mean() > 0.5
    per_prefix = lambda t: t.reshape(B, -1)[same].double()  # noqa: E731
    for k in ("logq_tok", "logq_corr", "alpha", "logkappa", "logkappa_corr", "logkappa_ref",
              "weights", "expected_len", "row_stats"):
        a, b = per_prefix(first[k]), per_prefix(want[k])
        assert bool(((a - b).abs() <= 64 * 2.0 ** -23 * b.abs().clamp(min=1.0)).all()), k
    a, b = first["loss"][:-1][same].double(), want["loss"][:-1][same].double()
    assert bool(((a - b).abs() <= 64 * 2.0 ** -23 * b.abs().clamp(min=1.0)).all())


def _same_rows(few, many, copies, skip=()):
    """Every output of `few` equals that of each copy in `many`, bit for bit."""
    for k, a in few.items():
        if k in skip or not torch.is_tensor(a):
            continue
        b = many[k].reshape(copies, -1)
        for i in (0, copies // 2, copies - 1):
            assert torch.equal(b[i], a.reshape(-1)), k


@pytest.mark.parametrize("V,dtype,n", [(24576, "f32", 64), (50004, "f32", 64), (49152, "bf16", 64),
                                       (4104, "bf16", 128), (4099, "f32", 64)])
def test_few_rows_equal_many(vsd, V, dtype, n):
    """Few rows of at least 48 chunks take the deeper ring, and few rows are verified
    in one kernel; the same rows n times over the shallow ring and two kernels: the
    same results bit for bit."""
    from paper_2602_05774_gb300 import inputs
    K, D = 5, 2  # 10 rows; 640, or 1280 of short aligned ones
    p = inputs.linear_problem(1, K, D, V, dtype, "gauss", "cuda", seed=V)
    q = {k: (v.repeat(*([n] + [1] * (v.dim() - 1))) if torch.is_tensor(v) else v)
         for k, v in p.items()}
    prm = vsd.params(like=p["draft"], kl_weight=0.5)
    a, b = _call(vsd, p, 1.0, prm), _call(vsd, q, 1.0, prm)
    _same_rows(a, b, n, skip=("loss", "grad"))
    assert torch.equal(b["loss"][:n], a["loss"][:1].expand(n))
    assert torch.equal(b["grad"].view(n, -1)[n - 1], a["grad"].view(-1) / n)
    s, t = (vsd.sample_paths(x["draft"], x["u_draft"], K, D, 1.0) for x in (p, q))
    _same_rows(s, t, n)
    _same_rows(*(vsd.verify_paths(x["draft"], x["target"], y["tokens"], x["u_accept"],
                                  x["u_correct"], K, D, 1.0) for x, y in ((p, s), (q, t))), n)
    r = [dict(r=vsd.reference_logkappa(x["draft"], x["target"], x["draft"].shape[0] // D, D, 1.0))
         for x in (p, q)]
    _same_rows(*r, n)


@pytest.mark.parametrize("V,dtype", [(24580, "f32"), (98312, "bf16")])
def test_sampling_many_long_rows_equals_few(vsd, V, dtype):
    """More than eight rows per SM of at least 48 (float32) or 96 chunks are
    sampled through the deeper ring, fewer through the shallow one."""
    from paper_2602_05774_gb300 import inputs
    n = 24
    p = inputs.linear_problem(1, 64, 1, V, dtype, "gauss", "cuda", seed=V)
    s, t = (vsd.sample_paths(p["draft"].repeat(m, 1), p["u_draft"].repeat(m), 64, 1, 1.0)
            for m in (1, n))
    _same_rows(s, t, n)


@pytest.mark.parametrize("rule", [0, 1])
def test_few_trees_with_long_rows_equal_many(vsd, rule):
    from paper_2602_05774_gb300 import inputs
    V, n = 49160, 80
    p = {k: (v.cuda() if torch.is_tensor(v) else v)
         for k, v in inputs.tree_problem(1, 8, 3, 3, V, seed=5).items()}
    q = {k: (v.repeat(*([n] + [1] * (v.dim() - 1))) if torch.is_tensor(v) else v)
         for k, v in p.items()}
    f = lambda x: vsd.verify_tree(x["draft"], x["target"], x["parent"], x["tokens"],  # noqa: E731
                                  x["u_accept"], x["u_correct"], 1.0, rule=rule)
    _same_rows(f(p), f(q), n)
    if rule == 0:
        f = lambda x: vsd.tree_estep_mstep(x["draft"], x["target"], x["parent"],  # noqa: E731
                                           x["tokens"], x["u_accept"], x["u_correct"], 1.0)
        _same_rows(f(p), f(q), n, skip=("loss", "grad"))


@pytest.mark.parametrize("V,R,n,dtype", [
    (330000, 64, 4, "bf16"),   # 323 chunks: 64 rows persistent, 256 two kernels
    (300001, 64, 8, "bf16"),   # 293 chunks, not 16-byte aligned: 64 and 512 rows
    (361001, 8, 64, "f32"),    # 706 chunks, not aligned: 8 and 512 rows
    (232000, 320, 4, "bf16"),  # 227 chunks, no gradient: 320 rows two kernels, 1280 persistent
])
def test_long_rows_by_either_route(vsd, V, R, n, dtype):
    """Long rows run on the persistent kernel or as two kernels, by their number:
    a batch and the same batch n times over, on either side of the line, give
    the same results bit for bit."""
    from paper_2602_05774_gb300 import inputs
    K, D = 8, 1
    p = inputs.linear_problem(R // K, K, D, V, dtype, "gauss", "cuda", seed=V)
    q = {k: (v.repeat(*([n] + [1] * (v.dim() - 1))) if torch.is_tensor(v) else v)
         for k, v in p.items()}
    grad = R < 320
    prm = vsd.params(like=p["draft"], kl_weight=0.5 if grad else 0.0,
                     grad_dtype=torch.float32)
    a, b = (_call(vsd, x, 1.0, prm, grad=grad) for x in (p, q))
    _same_rows(a, b, n, skip=("loss", "grad"))
    assert torch.equal(b["loss"][:-1].view(n, -1)[n - 1], a["loss"][:-1])
    if grad:  # (a mean over n times the prefixes: an exact factor)
        assert torch.equal(a["grad"].view(-1) / n, b["grad"].view(n, -1)[n - 1])


@pytest.mark.parametrize("V,dtype", [(32000, "bf16"), (4099, "f32"), (80000, "bf16")])
def test_gradient_in_the_drafts_place(vsd, V, dtype):
    """The gradient may be written over the draft logits: the elements with sparse
    terms are read before their row is written (linear paths with top-K terms, in
    one and in several segments a row, and trees)."""
    from paper_2602_05774_gb300 import inputs
    B, K, D = 4, 8, 3
    p = inputs.linear_problem(B, K, D, V, dtype, "spiked", "cuda", seed=V)
    prm = vsd.params(like=p["draft"], kl_weight=0.5)
    want = _call(vsd, p, 1.0, prm)
    out = vsd.linear_outputs(B, K, D, V, "cuda", grad=False, kl=True)
    out["grad"] = p["draft"]
    _call(vsd, p, 1.0, prm, out=out)
    for k in want:
        assert torch.equal(out[k], want[k]), k
    q = {k: (v.cuda() if torch.is_tensor(v) else v)
         for k, v in inputs.tree_problem(B, 24, 4, 4, V, seed=6, dtype=dtype).items()}
    a = (q["draft"], q["target"], q["parent"], q["tokens"], q["u_accept"], q["u_correct"])
    want = vsd.tree_estep_mstep(*a, 1.0)
    import ctypes as C
    ws = vsd.new_workspace(vsd.layout(B, V=V, N=24, parent=q["parent"]), "cuda")
    loss = torch.empty(B + 1, device="cuda")
    st = vsd.TreeEmOutputs(**dict(loss=loss.data_ptr(), grad=q["draft"].data_ptr()))
    ptr = [t.data_ptr() for t in a]
    assert vsd.load().vsd_tree_estep_mstep(
        ptr[0], ptr[1], int(dtype == "bf16"), vsd.layout(B, V=V, N=24, parent=q["parent"]), 1.0,
        ptr[3], ptr[4], ptr[5], C.byref(vsd.params(like=q["draft"])), C.byref(st), ws.data_ptr(),
        ws.numel(), torch.cuda.current_stream().cuda_stream) == 0
    assert torch.equal(q["draft"], want["grad"]) and torch.equal(loss, want["loss"])
