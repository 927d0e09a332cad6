"""Every entry point captured in a CUDA graph: the kernels of a call are
programmatic dependents of one another, and a replay on other inputs in the same
buffers gives the plain call's results bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vsd():
    from paper_2602_05774_gb300 import build, vsd as v
    build.build_library()
    v.load()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    return v


def _cuda(p):
    return {k: (v.cuda() if torch.is_tensor(v) else v) for k, v in p.items()}


def _flat(o, name=""):
    if torch.is_tensor(o):
        return {name: o}
    items = o.items() if isinstance(o, dict) else enumerate(o)
    return {k: t for n, v in items if v is not None for k, t in _flat(v, "%s.%s" % (name, n)).items()}


def _linear(vsd, seed, V=4104, dtype="bf16", B=3, K=4, D=5):
    from paper_2602_05774_gb300 import inputs
    return _cuda(inputs.linear_problem(B, K, D, V, dtype, "gauss", seed=seed))


def _em(vsd, p, ws, **kw):
    return vsd.estep_mstep(p["draft"], p["target"], p["u_draft"], p["u_accept"], p["u_correct"],
                           p["K"], p["D"], 1.0, workspace=ws, **kw)


def _calls(vsd):
    from paper_2602_05774_gb300 import inputs

    def ws_of(p):
        V = p["draft"].shape[1]
        return vsd.new_workspace(vsd.layout(p["draft"].shape[0] // (p["K"] * p["D"]), p["K"],
                                            p["D"], V), "cuda")

    def steps(p, ws):
        a = vsd.sample_paths(p["draft"], p["u_draft"], p["K"], p["D"], 1.0, workspace=ws)
        b = vsd.verify_paths(p["draft"], p["target"], a["tokens"], p["u_accept"], p["u_correct"],
                             p["K"], p["D"], 1.0, workspace=ws)
        return a, b, vsd.weighted_loss_fwd_bwd(p["draft"], b, p["K"], p["D"], 1.0, workspace=ws)

    def tree(rule):
        return lambda p, ws: vsd.verify_tree(p["draft"], p["target"], p["parent"], p["tokens"],
                                             p["u_accept"], p["u_correct"], 1.0, workspace=ws,
                                             rule=rule)

    def head(p, ws):
        o = vsd.lmhead_estep_mstep(p["hidden"], p["weight"], p["target"], p["u_draft"],
                                   p["u_accept"], p["u_correct"], p["K"], p["D"], 1.0,
                                   workspace=ws, grad=False)
        return o, vsd.lmhead_backward(p["hidden"], p["weight"], o["draft_logits"], p["K"], p["D"],
                                      1.0, ws, prm=vsd.params(like=p["target"]))

    def head_in(s):
        p = _cuda(inputs.lmhead_problem(3, 4, 5, 1032, 264, "cpu", seed=s))
        p.update(K=4, D=5)
        return p

    tree_in = lambda s: _cuda(inputs.tree_problem(3, 20, 4, 4, 1000, seed=s))  # noqa: E731
    tree_ws = lambda p: vsd.new_workspace(  # noqa: E731
        vsd.layout(3, V=1000, N=20, parent=p["parent"]), "cuda")
    tree_em = lambda p, ws: vsd.tree_estep_mstep(  # noqa: E731
        p["draft"], p["target"], p["parent"], p["tokens"], p["u_accept"], p["u_correct"], 1.0,
        workspace=ws)
    ref = lambda p, ws: dict(r=vsd.reference_logkappa(p["draft"], p["target"], 12, 5, 1.0))  # noqa: E731
    kl = lambda p, ws: _em(vsd, p, ws, prm=vsd.params(like=p["draft"], kl_weight=0.5))  # noqa: E731
    return {
        "em": (lambda s: _linear(vsd, s), ws_of, kl),
        "em_unaligned": (lambda s: _linear(vsd, s, 4099, "f32"), ws_of, kl),
        "em_persistent": (lambda s: _linear(vsd, s, 600000, "f32", 1, 1, 4), ws_of,
                          lambda p, ws: _em(vsd, p, ws)),
        "steps": (lambda s: _linear(vsd, s), ws_of, steps),
        "reference": (lambda s: _linear(vsd, s), ws_of, ref),
        "tree": (tree_in, tree_ws, tree(vsd.TREE_INDEPENDENT)),
        "tree_sequential": (tree_in, tree_ws, tree(vsd.TREE_SEQUENTIAL)),
        "tree_em": (tree_in, tree_ws, tree_em),
        "head": (head_in, lambda p: vsd.new_workspace(vsd.layout(3, 4, 5, 1032), "cuda"), head),
    }


@pytest.mark.parametrize("name", ["em", "em_unaligned", "em_persistent", "steps", "reference",
                                  "tree", "tree_sequential", "tree_em", "head"])
def test_captured_call_replays_on_new_inputs(vsd, name):
    make, ws_of, call = _calls(vsd)[name]
    p, q = make(1), make(2)
    ws = ws_of(p)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        call(p, ws)  # (kernels loaded before the capture)
    torch.cuda.current_stream().wait_stream(s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = call(p, ws)
    for k, v in q.items():
        if torch.is_tensor(v):
            p[k].copy_(v)
    for _ in range(3):
        for t in _flat(got).values():
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert vsd.device_status(ws) == (0, 0)
        want = _flat(call(q, ws_of(q)))
        for k, t in _flat(got).items():
            assert torch.equal(t, want[k]), k
