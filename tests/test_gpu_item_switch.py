"""One launch per round: sequences of one to three chunks, so that work items follow one another closely in a CTA of the walk."""
import pytest
import torch

import paper_2608_28158_b200 as H
from parity_util import compare, kernels_of, oracle_subset, run_gpu
from test_gpu_parity import check
from workloads import make_forest, make_inputs

pytestmark = pytest.mark.gpu


def _forest(kids, grandkids):
    """Every leaf from a boundary of its own (no fans), its replayed tail and own part one, two or three chunks; `grandkids` of them carry
    a leaf of the next round."""
    fork = [64 * (i + 1) + 1 + i * 7 % 63 for i in range(kids)]
    own = [(64 - f % 64, 128 - f % 64, 1, 65, 130)[i % 5] for i, f in enumerate(fork)]
    for i in range(grandkids):
        own[i] = 150 + i % 40
    par, off, lens = [-1] + [0] * kids, [0] + fork, [64 * (kids + 2)] + own
    for i in range(grandkids):
        par.append(1 + i)
        off.append(own[i] - i % 20)
        lens.append((1, 64, 70)[i % 3])
    return make_forest([(par, off, lens)])


@pytest.mark.parametrize("kids,grandkids,heads", [(36, 0, 4), (37, 0, 4), (38, 0, 4), (20, 20, 4), (75, 0, 8), (1, 0, 600)])
def test_short_sequences_behind_one_another(kids, grandkids, heads):
    """Sequences of one, two or three chunks (64 and 128 rows exactly among them), through the walk: a round of fewer items than CTAs,
    of one less and of some more, several tiers, many roots behind one another.  Two runs give the same bits."""
    fo = _forest(kids, grandkids)
    inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 23, device="cuda")
    got = {}

    def run():
        got["plan"], got["out"] = run_gpu(fo, inp, flags=H.HARTS_FLAG_ROUND_LAUNCHES)

    names = kernels_of(run)
    assert "tc_bwd_kernel" in names and "chunk_bwd_kernel" not in names and "scan_kernel" not in names, names
    plan, rounds = got["plan"], got["out"]
    assert plan.n_rounds == (3 if grandkids else 2)
    pick = sorted({0, heads - 1})
    tok, ref = oracle_subset(fo, inp, [0], pick)
    check(compare(rounds, tok, pick, ref, rows=True), "bf16")
    _, again = run_gpu(fo, inp, flags=H.HARTS_FLAG_ROUND_LAUNCHES)
    for n in rounds:
        assert torch.equal(rounds[n], again[n]), n
