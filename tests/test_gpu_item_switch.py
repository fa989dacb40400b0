"""One launch per round: sequences of one to three chunks, so that work items follow one another closely in a CTA of the walk."""
import pytest
import torch

import paper_2608_28158_b200 as H
from parity_util import compare, oracle_subset, run_gpu
from test_gpu_parity import check
from workloads import make_forest, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kids,heads", [(1, 1), (36, 4), (37, 4), (38, 4), (75, 8)])
def test_short_sequences_behind_one_another(kids, heads):
    """Leaves whose replayed tail and own part make one, two or three chunks (64 and 128 rows exactly among them), two rounds: fewer
    (sequence, head) pairs than SMs, a last tier with few items, several tiers.  Two runs give the
    same bits."""
    fork = [64 + i * 7 % 64 for i in range(kids)]
    own = [(64 - f % 64, 128 - f % 64, 1, 65, 130)[i % 5] for i, f in enumerate(fork)]
    fo = make_forest([([-1] + [0] * kids, [0] + fork, [200] + own)])
    inp = make_inputs(fo.n_tokens, heads, 128, 128, "bf16", 23)
    plan, rounds = run_gpu(fo, inp, flags=H.HARTS_FLAG_ROUND_LAUNCHES)
    assert plan.n_rounds == 2
    pick = sorted({0, heads - 1})
    tok, ref = oracle_subset(fo, inp, [0], pick)
    check(compare(rounds, tok, pick, ref, rows=True), "bf16")
    _, again = run_gpu(fo, inp, flags=H.HARTS_FLAG_ROUND_LAUNCHES)
    for n in rounds:
        assert torch.equal(rounds[n], again[n]), n
