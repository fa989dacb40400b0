"""The cut dK / dV work of small attention problems: key tiles whose query tiles end at and around a unit's edges, with groups
wide enough for the cut, fewer partial sums than units would want (a small dq tensor), the same forests without a cut, and
which problems are cut."""
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

from oracle import attn_oracle as ao
from test_gpu_attn import SCALE, _backward, _check_backward, _forward, _rel, _setup
from workloads import make_forest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("root,kids", [(40, ()), (1024, ()), (1025, (64, 65)), (500, (1, 63, 129, 300)), (600, (130,) * 6)])
@pytest.mark.parametrize("Hq,Hkv", [(1, 1), (6, 2)])
def test_split_backward(root, kids, Hq, Hkv):
    n = len(kids)
    fo = make_forest([([-1] + [i // 2 for i in range(n)], [0] + [max(1, (root, *kids)[i // 2] - i) for i in range(n)], [root, *kids])])
    _check_backward(fo, Hq, Hkv, 7)


def _is_cut(fo, Hq, Hkv):
    inp, phys, index, rows = _setup(fo, Hq, Hkv, 7, True)
    o, lse = _forward(phys, index)
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        _backward(phys, index, o, lse)
        torch.cuda.synchronize()
    return any("split_kernel" in e.key for e in p.key_averages())


@pytest.mark.parametrize("root,kids", [(1024, ()), (1025, (64, 65)), (500, (1, 63, 129, 300)), (600, (130,) * 6)])
@pytest.mark.parametrize("Hq,Hkv", [(16, 1), (32, 2)])
def test_split_backward_of_wide_groups(root, kids, Hq, Hkv):
    """Against fp64 attention with the ancestor mask and its autograd (the per-token oracle takes 15 s at 32 heads)."""
    n = len(kids)
    fo = make_forest([([-1] + [i // 2 for i in range(n)], [0] + [max(1, (root, *kids)[i // 2] - i) for i in range(n)], [root, *kids])])
    assert _is_cut(fo, Hq, Hkv)
    inp, phys, index, rows = _setup(fo, Hq, Hkv, 7)
    got = _backward(phys, index, *_forward(phys, index))
    mask = torch.zeros(fo.n_tokens, fo.n_tokens, dtype=torch.bool)
    for t, path in enumerate(ao.paths(fo)):
        mask[t, torch.as_tensor(path)] = True
    q, k, v, dO = (inp[n].cuda().double().transpose(0, 1) for n in ("q", "k", "v", "dO"))
    x = [y.requires_grad_() for y in (q, k, v)]
    s = (x[0] @ x[1].repeat_interleave(Hq // Hkv, 0).transpose(1, 2) * SCALE).masked_fill(~mask.cuda(), float("-inf"))
    ((s.softmax(-1) @ x[2].repeat_interleave(Hq // Hkv, 0)) * dO).sum().backward()
    errs = [_rel(y[rows].double().cpu().numpy(), r.grad.transpose(0, 1).cpu().numpy()) for y, r in zip(got, x)]
    assert max(errs) <= 1e-2, errs


def test_even_work_is_not_cut():
    """Where the items are even, or little work, cutting them costs more than it gives: the prompt of an agentic tree, one of
    1,500 tokens, and many short trees take the plain kernels."""
    agentic = ([-1] + [0] * 4, [0] + [6000] * 4, [6000, 900, 700, 900, 500])
    assert not _is_cut(make_forest([agentic]), 16, 16)
    assert not _is_cut(make_forest([([-1], [0], [1500])]), 8, 2)
    assert not _is_cut(make_forest([([-1, 0, 0], [0, 600, 300], [600, 200, 100])] * 40), 8, 4)
