"""Calls from a thread that has made no CUDA call of its own yet (a worker thread of a training or serving program)."""
import threading

import pytest
import torch

import paper_2608_28158_b200 as H
from parity_util import plan_of, to_physical
from workloads import make_attn_inputs, make_forest, make_gk, make_inputs

pytestmark = pytest.mark.gpu
FOREST = make_forest([([-1, 0, 0], [0, 300, 200], [400, 130, 90])])


def _la():
    plan = plan_of(FOREST).upload()
    x = to_physical(plan, make_inputs(FOREST.n_tokens, 2, 128, 128, "bf16", 3))
    ws = H.Workspace(plan, 2, 128, 128, torch.bfloat16)
    out = {n: torch.empty_like(x[m]) for n, m in (("o", "v"), ("dq", "q"), ("dk", "k"), ("dv", "v"), ("dg", "g"))}
    return out, lambda st: H.run_fwd_bwd(plan, ws, x["q"], x["k"], x["v"], x["g"], x["dO"], out=out, stream=st)


def _gk():
    plan = plan_of(FOREST).upload()
    inp = make_inputs(FOREST.n_tokens, 2, 128, 128, "bf16", 3)
    inp["g"] = make_gk(FOREST.n_tokens, 2, 128, 3)
    x = to_physical(plan, inp)
    states, scratch = (torch.empty(b, dtype=torch.uint8, device="cuda") for b in H.harts_la_gk_workspace_bytes(plan.tables, 2, 128, 128, 1))
    slots = torch.empty(max(plan.n_slots, 1) * 2 * 128 * 128, device="cuda")
    out = {n: torch.empty_like(x[m]) for n, m in (("o", "v"), ("dq", "q"), ("dk", "k"), ("dv", "v"), ("dg", "g"))}

    def run(st):
        H.harts_la_gk_fwd(plan, 0, x["q"], x["k"], x["v"], x["g"], out["o"], slots, states, stream=st)
        H.harts_la_gk_bwd(plan, 0, x["q"], x["k"], x["v"], x["g"], x["dO"], out["dq"], out["dk"], out["dv"], out["dg"], states, scratch,
                          stream=st)
    return out, run


def _attn():
    x = {n: t.cuda() for n, t in make_attn_inputs(FOREST.n_tokens, 4, 2, 128, "bf16", 3).items()}
    index = H.harts_attn_index(FOREST.tree_node_ptr, FOREST.node_parent, FOREST.node_fork_off, FOREST.node_len).upload()
    out = dict(o=torch.empty_like(x["q"]), lse=torch.empty(FOREST.n_tokens, 4, device="cuda"), dq=torch.empty_like(x["q"]),
               dk=torch.empty_like(x["k"]), dv=torch.empty_like(x["v"]))
    delta = torch.empty(FOREST.n_tokens, 4, device="cuda")

    def run(st):
        H.harts_attn_fwd(index, x["q"], x["k"], x["v"], out["o"], out["lse"], 0.088, stream=st)
        H.harts_attn_bwd(index, x["q"], x["k"], x["v"], out["o"], out["lse"], x["dO"], out["dq"], out["dk"], out["dv"], delta, 0.088,
                         stream=st)
    return out, run


@pytest.mark.parametrize("make", [_la, _gk, _attn])
def test_first_call_of_a_thread(make):
    out, run = make()
    stream = torch.cuda.current_stream()
    run(stream)
    torch.cuda.synchronize()
    want = {n: x.clone() for n, x in out.items()}
    for x in out.values():
        x.zero_()
    torch.cuda.synchronize()
    errors = []

    def work():
        try:
            run(stream)
        except H.HartsError as e:
            errors.append(e)
    t = threading.Thread(target=work)
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for n in out:
        assert torch.equal(out[n], want[n]), n
