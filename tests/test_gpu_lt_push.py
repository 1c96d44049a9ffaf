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
