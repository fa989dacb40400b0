"""Edges of the host side's tables: runs of positions in the row grouping, and a tree that is wider than the planner's
walk over neighbours."""
import random
import tracemalloc

import numpy as np
import pytest

import paper_2608_28158_b200 as H
from oracle import mb_oracle as mo
from test_attn_host import _check as _check_index
from test_mb_plan import _lex_trajs, _plan
from test_plan_oracle import random_tree
from workloads import make_forest


def _runs(seed):
    rng = np.random.default_rng(seed)
    return np.concatenate([np.arange(a, a + n) for a, n in zip(rng.integers(0, 150, 60), rng.integers(1, 50, 60))])


@pytest.mark.parametrize("m", [
    [], [0], [199], list(range(200)), [7] * 40, list(range(199, -1, -1)), [3, 4, 5, 4, 5, 6, 5, 3], _runs(1), _runs(2),
    np.random.default_rng(3).integers(0, 200, 700)], ids=range(10))
def test_rows_are_grouped_in_position_order(m):
    m = np.asarray(m, np.int32)
    ptr, pos = H.harts_logp_csr(200, m)
    assert np.array_equal(ptr, np.concatenate([[0], np.cumsum(np.bincount(m, minlength=200))]))
    assert np.array_equal(pos, np.argsort(m, kind="stable"))
    for bad in (-1, 200, 2147483647):
        with pytest.raises(H.HartsError):
            H.harts_logp_csr(200, np.append(m, bad))


@pytest.mark.parametrize("leaves", [255, 258, 300])
def test_greedy_in_a_tree_wider_than_the_walk(leaves):
    rnd = random.Random(leaves)
    wide = ([-1] + [0] * leaves, [0] + [rnd.randint(1, 3) for _ in range(leaves)], [3] + [rnd.randint(1, 2) for _ in range(leaves)])
    fo = make_forest([wide, random_tree(rnd, 9, 12)])
    plan = _plan(fo, 1, 80)
    trajs = _lex_trajs(fo, plan)
    orders = mo.greedy_orders(trajs)
    for order, policy in ((1, 0), (3, 1)):
        got = list(zip(*(a.tolist() for a in plan.greedy_trace(order, policy))))
        assert got == mo.greedy_place(trajs, orders[order], 80, best_fit=policy == 0)


@pytest.mark.parametrize("lens", [[-100000000], [-1, 5], [0], [2147483647] * 40], ids=["negative", "one_negative", "empty", "huge"])
def test_attention_index_refuses_malformed_lengths(lens):
    """A node length that no forest can have is refused as such, whatever it says about the size of the tables: the buffer
    that is made before the lengths are checked stays small (40 nodes of 2^31 - 1 tokens would ask for 20 GB)."""
    n = len(lens)
    tracemalloc.start()
    with pytest.raises(H.HartsError):
        H.harts_attn_index([0, n], [-1] + [0] * (n - 1), [0] + [1] * (n - 1), lens)
    peak = tracemalloc.get_traced_memory()[1]
    tracemalloc.stop()
    assert peak < 16 << 20


def test_attention_index_beyond_the_first_guess():
    """A comb of 300 nodes in a row, a leaf off each: the ancestor and descendant lists need more words than the first buffer
    has, and the call is repeated with the size it asks for."""
    n = 300
    par = [-1] + [x for i in range(n - 1) for x in (2 * i, 2 * i)] + [2 * n - 2]
    fo = make_forest([(par, [0] + [1] * (2 * n - 1), [1] * (2 * n))])
    _check_index(fo, None)
    ix = H.harts_attn_index(fo.tree_node_ptr, fo.node_parent, fo.node_fork_off, fo.node_len)
    assert len(ix.host) > 4096 + 64 * 2 * n + 2 * n // 16


@pytest.mark.parametrize("call", [H.harts_attn_index, H.harts_conv_index, H.harts_la_expand, H.harts_la_plan])
def test_a_negative_node_count_is_an_error(call):
    with pytest.raises(H.HartsError):
        call([0, -5], [], [], [])


@pytest.mark.parametrize("n_seq,n_chunks,heads,chunks", [
    (5, 448, 64, True), (5, 449, 64, False), (5, 28672, 1, True), (5, 28673, 1, False),        # 28,672 items
    (10, 44, 64, True), (10, 44, 65, False),                                                   # 640 (sequence, head) pairs
    (32, 128, 5, True), (32, 127, 5, False), (32, 127, 4, True)])                              # four chunks a sequence, or 128 pairs
@pytest.mark.parametrize("sizes", [H.harts_la_workspace_bytes, H.harts_la_gk_workspace_bytes])
def test_which_problems_bring_the_room_of_the_chunk_parallel_path(sizes, n_seq, n_chunks, heads, chunks):
    """The rule that picks the path also sizes the workspace: states alone (and flags), or their gradients and <S, dS> besides."""
    tables = H.binding.Tables(chunk=64, n_rows=64 * n_chunks, n_seq=n_seq, n_chunks=n_chunks)
    states = n_chunks * heads * 128 * 128 * 2
    got = sizes(tables, heads, 128, 128, H.HARTS_BF16)[0] - states
    assert (got >= states + n_chunks * heads * 4 * 128 * 4) == chunks
    assert chunks or got < states // 2 + 4096
