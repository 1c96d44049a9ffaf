"""LT push with its smaller work items: slots of one pair to more than an item's worth, rows that split over
many items, both weight forms, passes on either side of the accumulate form's width limit."""
import numpy as np
import pytest

import oracle
import paper_2404_17059_gb300 as P
from paper_2404_17059_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def graph():
    return I.rmat(11, 12 << 11, graph_seed=17)  # rows from none to several hundred edges


@pytest.mark.parametrize("words", [1, 2, 15, 16, 17, 33, 64, 65])
@pytest.mark.parametrize("form", ["equal", "uneven"])
def test_work_items(graph, words, form):
    g = graph
    w = I.lt_weighted_cascade(g) if form == "equal" else I.lt_random(g, graph_seed=3)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, None, w)
    seeds = I.top_degree_seeds(g, 5)
    T = 64 * words - 7
    b = oracle.simulate_threads("lt", g, seeds, T, 8, level_counts_len=16, lt_weight=w)
    for kw in ({}, {"chunk_edges": 5}, {"graph": 1}):
        a = P.cnd_lt_simulate_ex(G, seeds, T, 8, edge_checks=True, level_counts_len=16, word_bits=64 * words,
                                 direction="push", **kw)
        assert np.array_equal(a.spread, b.spread) and np.array_equal(a.node_count, b.node_count)
        assert a.edge_checks == b.edge_checks and np.array_equal(a.level_counts, b.level_counts)


@pytest.mark.parametrize("form", ["equal", "uneven"])
def test_long_items_of_wide_passes(form):
    """A row of 6,000 edges as one requested item of 2,047 pairs: 12 M tasks, whose indices have to be divided
    exactly by the pair count."""
    n, words = 6002, 2047
    g = I.csr_from_edges(n, np.concatenate([np.zeros(n - 2, np.int64), np.arange(1, 40)]),
                         np.concatenate([np.arange(1, n - 1), np.full(39, n - 1)]))
    w = np.full(g.m, 1 << 31, dtype=np.uint32)  # a spoke follows the hub in half of the trials
    w[g.col == n - 1] = (1 << 32) // 40 if form == "equal" else np.arange(1, 40) << 21
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, None, w)
    T = 64 * words - 7
    a, b = (P.cnd_lt_simulate_ex(G, [0], T, 4, edge_checks=True, level_counts_len=4, word_bits=64 * words,
                                 direction="push", stats=2, chunk_edges=c) for c in (16384, 0))
    assert a.stats["passes"] == 1 and a.stats["lt_counters"] == (form == "equal")
    assert np.array_equal(a.spread, b.spread) and np.array_equal(a.node_count, b.node_count)
    assert a.edge_checks == b.edge_checks and np.array_equal(a.level_counts, b.level_counts)
    o = oracle.simulate_threads("lt", g, [0], 256, 4, level_counts_len=4, lt_weight=w)
    assert np.array_equal(a.spread[:256], o.spread)
