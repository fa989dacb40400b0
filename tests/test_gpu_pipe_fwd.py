"""The pipelined forward walk at its edges: both widths of state columns, both sides of its line, ends of sequences, slots."""
import numpy as np
import pytest
import torch

import paper_2608_28158_b200 as H
from parity_util import compare, oracle_subset, plan_of, rel_err, run_gpu, to_physical
from test_gpu_parity import check
from workloads import make_forest, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [(257, 256, 320), (64 * 9, 300, 5), (64 * 40 + 1, 64, 1), (1217, 193, 63, 64, 65)])
@pytest.mark.parametrize("heads", [64, 80])
def test_edges(lens, heads):
    """Last rows, whole chunks, a tail of one row, branches that replay 1 to 63 rows; 64 heads (one root: two slices of 64 columns) and
    80 (one CTA for all 128 columns): rows against the oracle, the same bits in one launch and round by round."""
    offs = [0] + [lens[0] - 1 - 50 * i for i in range(len(lens) - 1)]
    fo = make_forest([([-1] + [0] * (len(lens) - 1), offs, list(lens))])
    inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 41, device="cuda")
    plan, out = run_gpu(fo, inp)
    assert plan.n_chunks >= 4 * plan.n_seq and plan.n_seq * heads >= 192
    pick = [0, 1, heads - 1]
    tok, ref = oracle_subset(fo, inp, [0], pick)
    check(compare(out, tok, pick, ref, rows=True), "bf16")
    _, rounds = run_gpu(fo, inp, flags=H.HARTS_FLAG_ROUND_LAUNCHES)
    for n in out:
        assert torch.equal(out[n], rounds[n]), n


@pytest.mark.parametrize("heads", [47, 48])
def test_both_sides_of_the_line(heads):
    """Four sequences of four chunks and more: 188 pairs take the scan and the chunk kernel, 192 the pipelined walk."""
    fo = make_forest([([-1, 0, 0, 1], [0, 700, 301, 200], [900, 500, 300, 390])])
    inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 42, device="cuda")
    plan, out = run_gpu(fo, inp, backward=False)
    assert plan.n_seq == 4 and plan.n_chunks >= 16
    tok, ref = oracle_subset(fo, inp, [0], [0, heads - 1], backward=False)
    check(compare(out, tok, [0, heads - 1], ref, names=("o",), rows=True), "bf16")


@pytest.mark.parametrize("shift", [0, 4])
def test_slots_and_states_are_those_of_the_other_paths(shift):
    """Slots (also where the array starts off a 32-byte sector) and chunk states against the fp32 kernels, and the outputs of a call
    that brings no workspace."""
    fo = make_forest([([-1] + [0] * 6, [0] + [64 * i + 65 for i in range(6)], [64 * 20 + 9] + [256] * 6)])
    heads = 64
    inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 43, device="cuda")
    plan = plan_of(fo).upload()
    p = to_physical(plan, inp)
    assert plan.n_chunks >= 4 * plan.n_seq and plan.n_seq * heads >= 192 and plan.n_slots >= 5
    got = {}
    for name, flags in (("pipe", 0), ("fma", H.HARTS_FLAG_FMA_KERNELS)):
        ws = H.Workspace(plan, heads, 128, 128, torch.bfloat16, flags)
        n = plan.n_slots * heads * 128 * 128
        ws.slots = torch.full((n + 8,), float("nan"), device="cuda")[shift:shift + n]
        out = H.run_fwd_bwd(plan, ws, p["q"], p["k"], p["v"], p["g"], None, backward=False)
        H.harts_la_check(ws.dev_status)
        states = ws.chunk_states[:plan.n_chunks * heads * 128 * 128 * 2].view(torch.bfloat16)
        got[name] = (out["o"], ws.slots, states)
    for a, b in zip(got["pipe"], got["fma"]):
        assert rel_err(a.float().cpu().numpy(), b.float().cpu().numpy()) < 6e-3      # two bf16 roundings on either side
    o = torch.empty_like(p["v"])
    H.harts_la_fwd(plan, 0, p["q"], p["k"], p["v"], p["g"], o, ws.slots, None, 0, ws.dev_status)
    assert torch.equal(o, got["pipe"][0])


def test_decays_in_two_factors():
    """Off the diagonal a decay is the product of a row's and a column's factor: mild and steep gates, and resets inside a chunk, are as
    far from 64 bits as bf16 operands leave them."""
    heads = 64
    fo = make_forest([([-1, 0, 0], [0, 1000, 333], [1100, 330, 280])])
    for scale, reset in ((0.001, 0), (1.0, 0), (30.0, 0), (0.05, -3000.0)):
        inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 44)
        inp["g"] = inp["g"] * scale
        if reset:
            inp["g"][::37] = reset
        _, out = run_gpu(fo, inp, backward=False)
        tok, ref = oracle_subset(fo, inp, [0], [0, heads - 1], backward=False)
        errs = compare(out, tok, [0, heads - 1], ref, names=("o",))
        assert errs["o"] < 6e-3 and np.isfinite(out["o"].float().cpu().numpy()).all(), (scale, reset, errs)
