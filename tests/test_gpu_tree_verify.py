"""Tree verification where its blocks take different ways: deep accepted paths
(nodes with and without an accepted child), and leaf rows read with the others or
only where a bonus token needs them."""
import numpy as np
import pytest
import torch

from tests.parity import compare_tree

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vsd():
    from paper_2602_05774_gb300 import build, vsd as v
    build.build_library()
    v.load()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    return v


def _case(B, parent, V, seed, noise):
    """Spiked logits; each node's token among its parent row's 4 largest."""
    g = torch.Generator().manual_seed(seed)
    N = len(parent)
    draft = torch.randn(B * N, V, generator=g) * 3.0
    target = draft + noise * torch.randn(B * N, V, generator=g)
    parent = torch.tensor(parent, dtype=torch.int32).repeat(B, 1)
    top = draft.bfloat16().float().topk(4, dim=1).indices.to(torch.int32)
    rows = (torch.arange(B).view(B, 1) * N + parent.clamp(min=0).long()).view(-1)
    tokens = top[rows, torch.randint(0, 4, (B * N,), generator=g)].view(B, N)
    tokens[:, 0] = 0
    p = dict(draft=draft.bfloat16(), target=target.bfloat16(), parent=parent, tokens=tokens,
             u_accept=torch.rand(B, N, generator=g), u_correct=torch.rand(B, N, generator=g))
    return p, {k: v.cuda() for k, v in p.items()}


def _verify(vsd, p, stats=True, rule=0):
    B, N = p["parent"].shape
    ws = vsd.new_workspace(vsd.layout(B, V=p["draft"].shape[1], N=N, parent=p["parent"]), "cuda")
    out = vsd.verify_tree(p["draft"], p["target"], p["parent"], p["tokens"], p["u_accept"],
                          p["u_correct"], 1.0, workspace=ws, rule=rule,
                          out=vsd.tree_outputs(B, N, "cuda", stats))
    return out, vsd.device_status(ws)


CHAIN = [-1] + list(range(150))
COMB = [-1] + [n - 2 if n % 2 and n > 1 else n - 1 for n in range(1, 200)]  # a leaf at every node


@pytest.mark.parametrize("parent", [CHAIN, COMB])
@pytest.mark.parametrize("noise", [0.0, 0.02])  # every node accepted; a rejection now and then
def test_deep_accepted_paths(vsd, oracle, parent, noise):
    p, c = _case(3, parent, 72, 11, noise)
    f = lambda t: t.float().numpy()  # noqa: E731
    orc = oracle.tree(f(p["draft"]), f(p["target"]), 1.0, p["parent"].numpy(),
                      p["tokens"].numpy(), f(p["u_accept"]), f(p["u_correct"]))
    for stats in (True, False):
        got, status = _verify(vsd, c, stats)
        assert status == (0, 0)
        compare_tree(got, orc)
    if noise == 0.0:
        depth = np.zeros(len(parent), int)
        for n in range(1, len(parent)):
            depth[n] = depth[parent[n]] + 1
        assert (got["accept_len"].cpu().numpy() == depth.max()).all()


@pytest.mark.parametrize("rule", [0, 1])
@pytest.mark.parametrize("copies", [1, 100])  # 3 and 300 rows, fewer and more than SMs
def test_leaf_rows_early_and_late(vsd, rule, copies):
    """A root and two leaves, every node accepted, so the bonus token is drawn at
    the first leaf's row: the same token whether the row is read with the others
    (row statistics; few rows under the sequential rule) or when it is needed.  A
    leaf row that enters no result sets no status bit without row statistics."""
    _, c = _case(1, [-1, 0, 0], 4104, 3, 0.0)

    def run(bad, stats):
        q = {k: v.repeat(*([copies] + [1] * (v.dim() - 1))) for k, v in c.items()}
        if bad is not None:
            q["target"].view(copies, 3, -1)[:, bad, 7] = float("nan")
        return _verify(vsd, q, stats, rule)

    want, status = run(None, True)
    assert status == (0, 0) and (want["deepest"] == 1).all()
    row = torch.softmax(c["target"][1].double(), 0).cumsum(0)
    tok = int(torch.searchsorted(row, c["u_correct"][0, 1].double().cuda(), right=True))
    assert (want["bonus"] == tok).all()
    got, status = run(None, False)
    assert status == (0, 0)
    for k in got:
        assert torch.equal(got[k], want[k]), k
    got, status = run(2, False)  # the leaf that no output reads
    assert status == (0, 0) and torch.equal(got["bonus"], want["bonus"])
    assert run(2, True)[1] == (6, vsd.STATUS_BAD_ROW)
    for stats in (True, False):
        got, status = run(1, stats)
        assert status == (6, vsd.STATUS_BAD_ROW) and (got["bonus"] == -1).all()
