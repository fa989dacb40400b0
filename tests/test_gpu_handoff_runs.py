"""Hand-off gradients of short sequences, summed in runs of eight consumers: runs that a boundary's list begins, ends and crosses, a round
issued alone beside the whole call, and the row-wise error."""
import numpy as np
import pytest
import torch

import paper_2608_28158_b200 as H
from parity_util import compare, kernels_of, oracle_subset, run_gpu
from test_gpu_parity import check
from workloads import make_forest, make_inputs

pytestmark = pytest.mark.gpu


def _fan(sizes):
    """`sizes[i]` short branches from boundary i + 1 of the root, forking at different rows behind it."""
    par, off, lens = [-1], [0], [64 * (len(sizes) + 1) + 9]
    for i, n in enumerate(sizes):
        for k in range(n):
            par.append(0)
            off.append(64 * (i + 1) + 1 + (7 * k + i) % 63)
            lens.append(1 + (11 * k) % 70)
    return make_forest([(par, off, lens)])


@pytest.mark.parametrize("sizes,heads", [((8, 8, 8, 9), 150), ((1, 7, 8, 9, 16, 2), 128), ((3, 30, 1, 1, 5), 128), ((16, 24), 128)])
def test_runs(sizes, heads):
    """Lists that fit the runs of eight, straddle them, and lie several in one; enough (sequence, head) pairs that the runs are taken."""
    fo = _fan(sizes)
    inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 61, device="cuda")
    got = {}

    def run():
        got["plan"], got["out"] = run_gpu(fo, inp)

    names = kernels_of(run)
    plan, out = got["plan"], got["out"]
    assert "tc_bwd_kernel" in names and "handoff_reduce" in names
    assert plan.n_rounds == 2 and plan.n_chunks < 4 * plan.n_seq and sum(sizes) * heads >= 4 * 8 * 148
    pick = [0, heads - 1]
    tok, ref = oracle_subset(fo, inp, [0], pick)
    check(compare(out, tok, pick, ref, rows=True), "bf16")
    _, again = run_gpu(fo, inp)
    _, rounds = _round_by_round(fo, inp)
    for n in out:
        assert torch.equal(out[n], again[n]) and torch.equal(out[n], rounds[n]), n


def _round_by_round(fo, inp):
    """The backward one round a call: every sequence leaves its own gradient there."""
    from parity_util import plan_of, to_physical
    plan = plan_of(fo).upload()
    p = to_physical(plan, inp)
    heads = p["q"].shape[1]
    ws = H.Workspace(plan, heads, 128, 128, torch.bfloat16)
    out = {"o": torch.empty_like(p["v"]), "dq": torch.empty_like(p["q"]), "dk": torch.empty_like(p["k"]), "dv": torch.empty_like(p["v"]),
           "dg": torch.empty_like(p["g"])}
    H.harts_la_fwd(plan, 0, p["q"], p["k"], p["v"], p["g"], out["o"], ws.slots, ws.chunk_states, 0, ws.dev_status)
    for r in range(plan.n_rounds, 0, -1):
        H.harts_la_bwd(plan, r, p["q"], p["k"], p["v"], p["g"], p["dO"], out["dq"], out["dk"], out["dv"], out["dg"], ws.chunk_states, ws.scratch, 0,
                       ws.dev_status)
    H.harts_la_check(ws.dev_status)
    rows = torch.as_tensor(plan.row_of_token.astype(np.int64), device="cuda")
    return plan, {n: x[rows] for n, x in out.items()}
