"""Attention at the edges of its tiles: runs of keys and of queries that end one short of, at and one past a step of the products
(16 rows), half a tile (64) and a tile (128), forward and backward against fp64 attention with the ancestor mask."""
import pytest
import torch

import paper_2608_28158_b200 as H
from oracle import attn_oracle as ao
from test_gpu_attn import SCALE, _backward, _forward, _rel, _setup
from test_gpu_attn_split import _is_cut
from workloads import make_forest

pytestmark = pytest.mark.gpu


def _check(fo, Hq, Hkv):
    inp, phys, index, rows = _setup(fo, Hq, Hkv, 11)
    o, lse = _forward(phys, index)
    grads = _backward(phys, index, o, lse)
    mask = torch.zeros(fo.n_tokens, fo.n_tokens, dtype=torch.bool)
    for t, path in enumerate(ao.paths(fo)):
        mask[t, torch.as_tensor(path)] = True
    q, k, v, dO = (inp[n].cuda().double().transpose(0, 1) for n in ("q", "k", "v", "dO"))
    x = [y.requires_grad_() for y in (q, k, v)]
    s = (x[0] @ x[1].repeat_interleave(Hq // Hkv, 0).transpose(1, 2) * SCALE).masked_fill(~mask.cuda(), float("-inf"))
    ref = s.softmax(-1) @ x[2].repeat_interleave(Hq // Hkv, 0)
    (ref * dO).sum().backward()
    # bf16 operands, P and dS rounded to bf16: 2^-9 each, adding up to 3e-3 over a few hundred terms
    assert _rel(o[rows].double().cpu().numpy(), ref.detach().transpose(0, 1).cpu().numpy()) <= 5e-3
    assert (lse[rows].double().cpu() - s.detach().logsumexp(-1).transpose(0, 1).cpu()).abs().max() <= 2e-3
    errs = [_rel(y[rows].double().cpu().numpy(), r.grad.transpose(0, 1).cpu().numpy()) for y, r in zip(grads, x)]
    assert max(errs) <= 1e-2, errs


@pytest.mark.parametrize("edge", [16, 64, 128])
@pytest.mark.parametrize("Hq,Hkv", [(2, 2), (3, 1)])
def test_runs_around_a_tile_edge(edge, Hq, Hkv):
    """A root and two levels of branches whose lengths lie around the edge; every branch forks inside its parent too."""
    for d in (-1, 0, 1):
        n = 128 + edge + d
        lens = [n, edge + d, edge, edge + 1, 2 * edge + d]
        _check(make_forest([([-1, 0, 0, 1, 1], [0, n, edge + d, edge + d, max(1, edge // 2)], lens)]), Hq, Hkv)


@pytest.mark.parametrize("root,Hq,Hkv,cut", [(300, 2, 2, False), (1500, 16, 1, True)])
def test_dq_over_o(root, Hq, Hkv, cut):
    """dq is work memory until its values are written, and may be o's memory: the gradients are those of a call with memory of its own,
    row by row, whole and cut."""
    fo = make_forest([([-1, 0, 0], [0, root, root // 2], [root, 130, 70])])
    inp, phys, index, rows = _setup(fo, Hq, Hkv, 12)
    assert _is_cut(fo, Hq, Hkv) == cut
    o, lse = _forward(phys, index)
    want = _backward(phys, index, o, lse)
    dk, dv = torch.empty_like(phys["k"]), torch.empty_like(phys["v"])
    delta = torch.empty_like(lse)
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    H.harts_attn_bwd(index, phys["q"], phys["k"], phys["v"], o, lse, phys["dO"], o, dk, dv, delta, SCALE, dev_status=status)
    H.harts_la_check(status)
    for a, b in zip((o, dk, dv), want):
        assert torch.equal(a, b)
