"""The chunk-parallel linear-attention path at its edges and at the line where the walk kernels take over."""
import numpy as np
import pytest
import torch

import paper_2608_28158_b200 as H
from oracle import gk_oracle as go
from oracle import la_oracle as lo
from parity_util import compare, oracle_subset, plan_of, rel_err, run_gpu, to_physical
from test_gpu_parity import check
from workloads import make_forest, make_gk, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [(1,), (63,), (64,), (65, 1), (129, 64, 63), (64 * 40 + 1, 64, 1)])
def test_chunk_parallel_edges(lens):
    """One row, one row short of and past a chunk, single-chunk sequences, a boundary exported by the last chunk but one --
    in every width of the scan's state slices (1, 50 and 100 heads: 32, 64 and 128 columns)."""
    fo = make_forest([([-1] + [0] * (len(lens) - 1), [0] + [lens[0]] * (len(lens) - 2) + [max(1, lens[0] - 1)] * (len(lens) > 1), list(lens))])
    for heads in (1, 50, 100):
        inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 31)
        plan, out = run_gpu(fo, inp)
        pick = [0, heads - 1] if heads > 1 else [0]
        tok, ref = oracle_subset(fo, inp, [0], pick)
        check(compare(out, tok, pick, ref, rows=True), "bf16")


@pytest.mark.parametrize("lens", [(1,), (63,), (64,), (65, 1), (129, 64, 63), (64 * 20 + 1, 64, 1)])
def test_fp32_edges(lens):
    """The same edges through the fp32 kernels (d = 64); 20 chunks exceed the sums one walking thread keeps in flight."""
    fo = make_forest([([-1] + [0] * (len(lens) - 1), [0] + [lens[0]] * (len(lens) - 2) + [max(1, lens[0] - 1)] * (len(lens) > 1), list(lens))])
    inp = make_inputs(fo.n_tokens, 3, 64, 64, "fp32", 32)
    plan, out = run_gpu(fo, inp)
    tok, ref = oracle_subset(fo, inp, [0], [0, 1, 2])
    check(compare(out, tok, [0, 1, 2], ref, rows=True), "fp32")


@pytest.mark.parametrize("heads", [63, 64])
def test_both_sides_of_the_chunk_parallel_line(heads):
    """454 chunks x 63 heads take the chunk-parallel path, x 64 the walk kernels in their one-launch form: both against the
    oracle, and bit-equal to one launch per round."""
    fo = make_forest([([-1, 0, 0, 1], [0, 14000, 6001, 4000], [14000, 8000, 3000, 3901])])
    inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 12, device="cuda")
    plan, out = run_gpu(fo, inp)
    assert (plan.n_chunks * heads <= 28672) == (heads == 63), plan.n_chunks
    tok, ref = oracle_subset(fo, inp, [0], [0, heads - 1])
    check(compare(out, tok, [0, heads - 1], ref, rows=True), "bf16")
    _, rounds = run_gpu(fo, inp, flags=H.HARTS_FLAG_ROUND_LAUNCHES)
    for n in out:
        assert torch.equal(out[n], rounds[n]), n


@pytest.mark.parametrize("heads", [64, 65])
def test_both_sides_of_the_chain_line(heads):
    """Ten sequences of four or more chunks: 640 (sequence, head) pairs take the chunk-parallel path, 650 the walk."""
    fo = make_forest([([-1] + [0] * 9, [0] + [256] * 9, [512] + [270] * 9)])
    inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 13, device="cuda")
    plan, out = run_gpu(fo, inp)
    assert plan.n_seq == 10 and plan.n_chunks >= 40
    tok, ref = oracle_subset(fo, inp, [0], [0, heads - 1])
    check(compare(out, tok, [0, heads - 1], ref, rows=True), "bf16")
    _, rounds = run_gpu(fo, inp, flags=H.HARTS_FLAG_ROUND_LAUNCHES)
    for n in out:
        assert torch.equal(out[n], rounds[n]), n


def test_fp32_more_items_than_resident_blocks():
    """460 chunks x 2 heads: every kernel's CTAs take several items in turn, in one call and round by round."""
    fo = make_forest([([-1, 0, 0, 1], [0, 14000, 6001, 4000], [14000, 8000, 3000, 4333])])
    inp = make_inputs(fo.n_tokens, 2, 64, 64, "fp32", 14)
    plan, out = run_gpu(fo, inp)
    assert plan.n_chunks * 2 > 6 * torch.cuda.get_device_properties(0).multi_processor_count
    tok, ref = oracle_subset(fo, inp, [0], [0, 1])
    check(compare(out, tok, [0, 1], ref, rows=True), "fp32")
    _, rounds = run_gpu(fo, inp, flags=H.HARTS_FLAG_ROUND_LAUNCHES)
    for n in out:
        assert torch.equal(out[n], rounds[n]), n


def test_fp32_call_for_one_sequence_does_not_pay_for_the_forest():
    """A packed call names a range of sequences: one sequence of one chunk takes about as long beside 6,000 chunks x 8 heads as
    beside two (a grid of the whole forest's items made it 3 times as long)."""
    def median_us(root):
        fo = make_forest([([-1, 0], [0, root], [root + 64, 64])])
        plan = plan_of(fo).upload()
        x, g = torch.zeros(fo.n_tokens, 8, 64, device="cuda"), torch.zeros(fo.n_tokens, 8, device="cuda")
        o, ws, n = torch.empty_like(x), H.Workspace(plan, 8, 64, 64, torch.float32), plan.n_seq
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(52)]
        for e in ev:
            H.harts_la_fwd_seqs(plan.tables, n - 1, n, x, x, x, g, o, ws.slots, ws.chunk_states, 0, ws.dev_status)
            e.record()
        torch.cuda.synchronize()
        H.harts_la_check(ws.dev_status)
        return sorted(a.elapsed_time(b) * 1e3 for a, b in zip(ev[1:-1], ev[2:]))[25]

    few, many = median_us(128), median_us(64 * 6000)
    print(f"one sequence: {few:.1f} us beside 2 chunks, {many:.1f} us beside 6,000")
    assert many < 1.75 * few


@pytest.mark.parametrize("name", ["q", "k", "v", "dO"])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_fp32_non_finite_rows_keep_to_the_causal_side(name, bad):
    """An infinity or NaN in one row must not reach what does not depend on it: outputs and dq of the rows before it (k, v), dk and
    dv of the rows after it (q, dO), bit for bit -- wherever the row stands in its chunk."""
    fo = make_forest([([-1], [0], [200])])
    inp = make_inputs(fo.n_tokens, 2, 64, 64, "fp32", 16)
    _, clean = run_gpu(fo, inp)
    for t in (1, 6, 37, 63, 64, 127, 130, 198):
        x = {n: y.clone() for n, y in inp.items()}
        x[name][t, 0] = bad
        _, out = run_gpu(fo, x)
        for n in ("o", "dq") if name in "kv" else ("dk", "dv"):
            rows = slice(0, t) if name in "kv" else slice(t + 1, None)
            assert torch.equal(out[n][rows], clean[n][rows]), (n, t)
            assert torch.equal(out[n][:, 1], clean[n][:, 1]), (n, t)


@pytest.mark.parametrize("reset", [-100.0, -3000.0])
def test_fp32_keeps_its_precision_behind_steep_gates(reset):
    """One token in a hundred forgets everything before it.  The running log-decay of a chunk is large from there on, and the
    decay between two later rows is the exponential of a difference of two such sums: in 32 bits it was off by 2^-24 of the
    sums (8e-5 at -3000).  64-term fp32 sums are off by at most 64 * 2^-24."""
    fo = make_forest([([-1, 0, 0], [0, 700, 333], [700, 300, 250])])
    inp = make_inputs(fo.n_tokens, 2, 64, 64, "fp32", 17)
    gen = torch.Generator().manual_seed(17)
    inp["g"] = torch.where(torch.rand(inp["g"].shape, generator=gen) < 0.01, torch.tensor(reset), inp["g"])
    _, out = run_gpu(fo, inp)
    tok, ref = oracle_subset(fo, inp, [0], [0, 1])
    errs = compare(out, tok, [0, 1], ref)
    assert all(e <= 64 * 2.0 ** -24 for e in errs.values()), errs


def _gk_dg(fo, inp):
    plan = plan_of(fo).upload()
    x = to_physical(plan, inp)
    n, heads, d = x["q"].shape
    states, scratch = (torch.empty(b, dtype=torch.uint8, device="cuda") for b in H.harts_la_gk_workspace_bytes(plan.tables, heads, d, d, 1))
    slots, status = torch.empty(max(plan.n_slots, 1) * heads * d * d, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda")
    o, dq, dk, dv, dg = (torch.empty_like(x[m]) for m in ("v", "q", "k", "v", "g"))
    H.harts_la_gk_fwd(plan, 0, x["q"], x["k"], x["v"], x["g"], o, slots, states, 0, status)
    H.harts_la_gk_bwd(plan, 0, x["q"], x["k"], x["v"], x["g"], x["dO"], dq, dk, dv, dg, states, scratch, 0, status)
    H.harts_la_check(status)
    return dg[torch.as_tensor(plan.row_of_token.astype(np.int64), device="cuda")]


@pytest.mark.parametrize("gates", [1.0, 0.0])
@pytest.mark.parametrize("form", ["scalar", "per_channel"])
def test_dg_is_as_exact_as_in_the_walk(form, gates):
    """Seven sequences x 4 heads take the chunk-parallel path, the same four heads 24 times over the walk kernels.  Both hold the
    boundary gradient in 32 bits where dg needs it: against the oracle the one is not further off than the other (without decay
    a bf16 gradient made it 1.4 times as far)."""
    fo = make_forest([([-1] + [0] * 6, [0] + [700] * 6, [900] + [330] * 6)])
    inp = make_inputs(fo.n_tokens, 4, 128, 128, "bf16", 18)
    if form == "per_channel":
        inp["g"] = make_gk(fo.n_tokens, 4, 128, 18)
    inp["g"] = inp["g"] * gates
    many = {n: x.repeat(1, 24, *[1] * (x.dim() - 2)) for n, x in inp.items()}
    oracle, run = (go, _gk_dg) if form == "per_channel" else (lo, lambda fo, x: run_gpu(fo, x)[1]["dg"])
    ref = oracle.forest_eval(fo, *(inp[n] for n in ("q", "k", "v", "g", "dO")))["dg"]
    chunk, walk = (rel_err(run(fo, x)[:, :4].cpu().numpy(), ref) for x in (inp, many))
    print(f"{form} x{gates}: dg error {chunk:.2e} chunk-parallel, {walk:.2e} walk")
    assert chunk <= 1.1 * walk
