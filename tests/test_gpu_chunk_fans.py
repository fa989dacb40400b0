"""Fans of short branches through the chunk-parallel path: both sides of its line, and slots exported by one chunk after another."""
import numpy as np
import pytest
import torch

import paper_2608_28158_b200 as H
from oracle import gk_oracle as go
from parity_util import compare, kernels_of, oracle_subset, rel_err, row_err, run_gpu
from test_gpu_gk import check as check_gk, make_gk, run_gk
from test_gpu_parity import check
from workloads import make_forest, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads", [36, 37])
def test_both_sides_of_the_line_of_fans(heads):
    """32 sequences of fewer than four chunks: 1,152 (sequence, head) pairs take the chunk-parallel path, 1,184 the walk."""
    fo = make_forest([([-1] + [0] * 31, [0] + [1 + 4 * i for i in range(31)], [130] + [2 * i + 1 for i in range(31)])])
    inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 13, device="cuda")
    plan, out = run_gpu(fo, inp)
    assert plan.n_seq == 32 and plan.n_chunks < 4 * plan.n_seq
    tok, ref = oracle_subset(fo, inp, [0], [0, heads - 1])
    check(compare(out, tok, [0, heads - 1], ref, rows=True), "bf16")
    _, rounds = run_gpu(fo, inp, flags=H.HARTS_FLAG_ROUND_LAUNCHES)
    for n in out:
        assert torch.equal(out[n], rounds[n]), n


def _slots_in_a_row():
    """Two short branches from each of seven consecutive chunks."""
    forks = [64 * (i // 2 + 1) + 1 + 4 * i for i in range(14)]
    return make_forest([([-1] + [0] * 14, [0] + forks, [64 * 9 + 6] + [5 + i for i in range(14)])])


@pytest.mark.parametrize("heads,columns", [(1, 32), (40, 64), (75, 128)])
def test_a_slot_from_every_chunk(heads, columns):
    """Forks in each of seven consecutive chunks, the scan over 32, 64 and 128 columns of state at a time: slots are published in turn."""
    fo = _slots_in_a_row()
    inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 17, device="cuda")
    got = {}

    def run():
        got["plan"], got["out"] = run_gpu(fo, inp)

    names = kernels_of(run)
    assert "chunk_fwd_kernel" in names and f"scan_kernel<false, {columns}, false>" in names, names
    assert got["plan"].n_slots == 7
    pick = sorted({0, heads - 1})
    tok, ref = oracle_subset(fo, inp, [0], pick)
    check(compare(got["out"], tok, pick, ref, rows=True), "bf16")


@pytest.mark.parametrize("heads,columns", [(1, 64), (75, 128)])
def test_a_slot_from_every_chunk_per_channel(heads, columns):
    fo = _slots_in_a_row()
    got = {}

    def run():
        got["plan"], got["out"] = run_gk(fo, heads, 128, "bf16", 18, raw=True)

    names = kernels_of(run)
    assert "gk_chunk_fwd_kernel" in names and f"scan_kernel<false, {columns}, true>" in names, names
    assert got["plan"].n_slots == 7
    inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 18)
    inp["g"] = make_gk(fo.n_tokens, heads, 128, 18)
    pick = sorted({0, heads - 1})
    one = {n: x[:, pick].contiguous() for n, x in inp.items()}
    ref = go.forest_eval(fo, one["q"], one["k"], one["v"], one["g"], one["dO"])
    errs = {}
    for n, x in got["out"].items():
        errs[n], errs[n + ".row"] = rel_err(x[:, pick], ref[n]), row_err(x[:, pick], ref[n])
    check_gk(errs, "bf16")


@pytest.mark.parametrize("kids", [33, 70])
@pytest.mark.parametrize("gk", [False, True])
def test_a_boundary_with_many_consumers(kids, gk):
    """One boundary that more than 32 (64) sequences start from: their flags are looked at 32 at a time, their gradients summed in
    table order, with the same bits in one launch and round by round."""
    fo = make_forest([([-1] + [0] * kids, [0] + [64 + 1 + i % 60 for i in range(kids)], [130] + [1 + i % 7 for i in range(kids)])])
    if gk:
        plan, errs = run_gk(fo, 2, 128, "bf16", 19)
        check_gk(errs, "bf16")
        (_, out), (_, rounds) = (run_gk(fo, 2, 128, "bf16", 19, raw=True, flags=f) for f in (0, H.HARTS_FLAG_ROUND_LAUNCHES))
    else:
        inp = make_inputs(fo.n_tokens, 2, 128, 128, "bf16", 19)
        plan, out = run_gpu(fo, inp)
        tok, ref = oracle_subset(fo, inp, [0], [0, 1])
        check(compare(out, tok, [0, 1], ref, rows=True), "bf16")
        _, rounds = run_gpu(fo, inp, flags=H.HARTS_FLAG_ROUND_LAUNCHES)
    assert max(np.diff(plan.slot_cons_ptr)) >= kids - 1
    for n in out:
        assert np.array_equal(np.asarray(torch.as_tensor(out[n]).float().cpu()), np.asarray(torch.as_tensor(rounds[n]).float().cpu())), n
