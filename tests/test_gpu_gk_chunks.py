"""Edges of the chunk-parallel per-channel-decay path (one work item per chunk and head, states in memory) against the
oracle: sequences of one row, around a chunk's 64 rows, replayed rows, one or many items per CTA, gates mild enough for
the dense diagonal blocks and steep enough for the exact ones."""
import pytest

from test_gpu_gk import check, run_gk
from workloads import make_forest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("strong_every", [0, 3])
@pytest.mark.parametrize("heads", [1, 3])
@pytest.mark.parametrize("lens", [(1,), (63,), (64,), (65, 1), (129, 64, 63), (300, 17, 200)])
def test_edges(lens, heads, strong_every):
    n = len(lens)
    fo = make_forest([([-1] + [0] * (n - 1), [0] + [lens[0]] * (n - 2) + [max(1, lens[0] - 1)] * (n > 1), list(lens))])
    _, errs = run_gk(fo, heads, 128, "bf16", 7, strong_every=strong_every, strong_shift=60.0)
    check(errs, "bf16")


def test_more_items_than_resident_blocks():
    fo = make_forest([([-1, 0, 0], [0, 640, 333], [640, 300, 200])])
    plan, errs = run_gk(fo, 32, 128, "bf16", 9)
    assert plan.n_chunks * 32 > 2 * 148
    check(errs, "bf16")
