"""The LM head's backward on CTA pairs from a gradient in scratch memory, at the
edges of its tiles (256 x 256, K blocks of 64, the last tiles' K shared by two
pairs), and without scratch (the gradient made on chip): every output within
the fp32 summation bound K 2^-24 sum |a_k b_k| of the float64 product of the
written bf16 gradient."""
import ctypes as C

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


SHAPES = [  # B, K, D, V, H
    (1, 1, 1, 8, 8),          # one row
    (1, 5, 1, 264, 136),
    (3, 17, 5, 520, 264),     # R = 255
    (2, 16, 8, 1032, 256),    # R = 256, H = one tile
    (1, 257, 1, 72, 520),     # R = 257 would need K > 256: see below
    (20, 16, 8, 264, 2056),   # d_hidden: 10 x 9 tiles, whole ones and shared ones
]


@pytest.mark.parametrize("scratch", [True, False])
@pytest.mark.parametrize("B,K,D,V,H", SHAPES)
def test_backward_tiles_within_bound(vsd, B, K, D, V, H, scratch):
    from paper_2602_05774_gb300 import inputs
    if K > 256:
        B, K = K, 1  # R = 257 as prefixes
    R = B * K * D
    p = inputs.lmhead_problem(B, K, D, V, H, "cuda", seed=V + H)
    x = inputs.linear_problem(B, K, D, V, "bf16", "gauss", "cuda", seed=R)
    ws = vsd.new_workspace(vsd.layout(B, K, D, V), "cuda")
    prm = vsd.params(like=x["draft"])
    fw = vsd.estep_mstep(x["draft"], x["target"], x["u_draft"], x["u_accept"], x["u_correct"], K,
                         D, 1.0, prm=prm, workspace=ws)
    G, h, w = fw["grad"].double(), p["hidden"].double(), p["weight"].double()
    if scratch:
        bw = vsd.lmhead_backward(p["hidden"], p["weight"], x["draft"], K, D, 1.0, ws, prm=prm)
    else:
        bw = dict(d_hidden=torch.empty(R, H, device="cuda"),
                  d_weight=torch.empty(V, H, device="cuda"))
        ptr = lambda t: C.c_void_p(t.data_ptr())  # noqa: E731
        code = vsd.load().vsd_lmhead_backward(
            ptr(p["hidden"]), ptr(p["weight"]), H, ptr(x["draft"]), vsd.layout(B, K, D, V), 1.0,
            C.byref(prm), ptr(bw["d_hidden"]), ptr(bw["d_weight"]), ptr(ws), ws.numel(),
            C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert code == 0
    torch.cuda.synchronize()
    assert vsd.device_status(ws) == (0, 0)
    for name, a, b in (("d_hidden", G, w), ("d_weight", G.t(), h)):
        bound = a.shape[1] * 2.0 ** -24 * (a.abs() @ b.abs()) + 1e-30
        err = (bw[name].double() - a @ b).abs()
        assert bool((err <= bound).all()), "%s off by %g" % (name, float((err - bound).max()))


# few rows: one tile, several a CTA; pairs: one tile, a chunk, two units
@pytest.mark.parametrize("M,N", [(1, 8), (128, 40008), (129, 8), (256, 1024), (300, 1032)])
# K blocks: around the rings' four and six stages; 33: few tiles of few rows on pairs
@pytest.mark.parametrize("kb", [1, 2, 4, 5, 6, 7, 12, 13, 33])
def test_every_commit_is_waited_for(vsd, M, N, kb):
    """The pair leaves once the arrivals of its last commits have landed, at
    fewer K blocks than a ring has stages, as many, and more; a wait for a
    phase that never comes would show as its 2 s limit.  Inputs whose partial
    sums are exact in float32: the float64 product, rounded once."""
    K = 64 * kb - 8
    g = torch.Generator(device="cuda").manual_seed(K + M)
    h = torch.randint(-2, 3, (M, K), generator=g, device="cuda").bfloat16()
    w = (torch.randint(-64, 65, (N, K), generator=g, device="cuda").float() / 256).bfloat16()
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    vsd.lmhead_logits(h, w, workspace=ws)
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    a.record()
    got = [vsd.lmhead_logits(h, w, workspace=ws) for _ in range(4)]
    b.record()
    torch.cuda.synchronize()
    assert vsd.device_status(ws) == (0, 0)
    assert a.elapsed_time(b) < 500
    want = (h.double() @ w.double().t()).bfloat16()
    for x in got:
        assert torch.equal(x, want)


@pytest.mark.parametrize("R,V,H", [(16, 40, 64), (128, 168, 520), (300, 1032, 136)])
def test_backward_on_chip_waits_for_its_commits(vsd, R, V, H):
    """Without scratch, at few and many K blocks per tile and several tiles: no
    wait at the end of the kernel is for a phase that never comes (2 s)."""
    from paper_2602_05774_gb300 import inputs
    p = inputs.lmhead_problem(R, 1, 1, V, H, "cuda", seed=V)
    x = inputs.linear_problem(R, 1, 1, V, "bf16", "gauss", "cuda", seed=V)
    ws = vsd.new_workspace(vsd.layout(R, 1, 1, V), "cuda")
    prm = vsd.params(like=x["draft"])
    vsd.estep_mstep(x["draft"], x["target"], x["u_draft"], x["u_accept"], x["u_correct"], 1, 1,
                    1.0, prm=prm, workspace=ws)
    dh, dw = torch.empty(R, H, device="cuda"), torch.empty(V, H, device="cuda")
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    for ev in (a, b):  # (the first call loads the kernels)
        assert vsd.load().vsd_lmhead_backward(
            p["hidden"].data_ptr(), p["weight"].data_ptr(), H, x["draft"].data_ptr(),
            vsd.layout(R, 1, 1, V), 1.0, C.byref(prm), dh.data_ptr(), dw.data_ptr(),
            ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream) == 0
        ev.record()
    torch.cuda.synchronize()
    assert vsd.device_status(ws) == (0, 0) and a.elapsed_time(b) < 500


def test_backward_scratch_is_the_callers_choice(vsd):
    """scratch=False holds no dense gradient (its R*V bf16 values would dominate
    here) and gives the bits of the call without scratch; a tensor is used as it
    is and gives those of the default."""
    from paper_2602_05774_gb300 import inputs
    B, K, D, V, H = 16, 8, 4, 32008, 64
    R = B * K * D
    p = inputs.lmhead_problem(B, K, D, V, H, "cuda", seed=9)
    x = inputs.linear_problem(B, K, D, V, "bf16", "gauss", "cuda", seed=9)
    ws = vsd.new_workspace(vsd.layout(B, K, D, V), "cuda")
    vsd.estep_mstep(x["draft"], x["target"], x["u_draft"], x["u_accept"], x["u_correct"], K, D,
                    1.0, workspace=ws, grad=False)
    dh, dw = torch.empty(R, H, device="cuda"), torch.empty(V, H, device="cuda")

    def run(scratch):
        dh.fill_(float("nan")), dw.fill_(float("nan"))
        torch.cuda.synchronize()
        torch.cuda.reset_peak_memory_stats()
        before = torch.cuda.memory_allocated()
        vsd.lmhead_backward(p["hidden"], p["weight"], x["draft"], K, D, 1.0, ws, d_hidden=dh,
                            d_weight=dw, scratch=scratch)
        torch.cuda.synchronize()
        held = torch.cuda.max_memory_allocated() - before
        return dh.clone(), dw.clone(), held

    *default, held = run(True)
    assert held >= 2 * R * V
    *chip, held = run(False)
    assert held == 0
    buf = torch.full((R * V,), float("nan"), dtype=torch.bfloat16, device="cuda")
    *given, held = run(buf)
    assert held == 0 and torch.isfinite(buf).all()
    for a, b in zip(default, given):
        assert torch.equal(a, b)
    dh2, dw2 = torch.empty_like(dh), torch.empty_like(dw)
    prm = vsd.params(like=x["draft"])
    assert vsd.load().vsd_lmhead_backward(
        p["hidden"].data_ptr(), p["weight"].data_ptr(), H, x["draft"].data_ptr(),
        vsd.layout(B, K, D, V), 1.0, C.byref(prm), dh2.data_ptr(), dw2.data_ptr(), ws.data_ptr(),
        ws.numel(), torch.cuda.current_stream().cuda_stream) == 0
    assert torch.equal(chip[0], dh2) and torch.equal(chip[1], dw2)
    with pytest.raises(ValueError):
        run(buf[:-1])
