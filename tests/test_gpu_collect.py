"""Frontier collect of passes of more than four dirty-mask words: word counts at the edges of a mask word and
of the groups of 128 words a warp goes over, both models' counting forms, host-driven and captured calls."""
import numpy as np
import pytest

import oracle
import paper_2404_17059_gb300 as P
from paper_2404_17059_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def graph():
    g = I.rmat(10, 9 << 10, graph_seed=21)
    p = I.ic_uniform_random(g, 0.25, graph_seed=21)
    w = I.lt_weighted_cascade(g)
    return g, p, w, P.cnd_graph_create(g.n, g.row_ptr, g.col, p, w)


@pytest.mark.parametrize("words", [256, 257, 319, 320, 321, 383, 385, 2048])
@pytest.mark.parametrize("model", ["ic", "lt"])
@pytest.mark.parametrize("captured", [0, 1])
def test_wide_pass(graph, words, model, captured):
    g, p, w, G = graph
    T = 64 * words - 5
    seeds = I.uniform_seeds(g.n, 3, words)
    fn = P.cnd_ic_simulate_ex if model == "ic" else P.cnd_lt_simulate_ex
    kw = {"ic_prob": p} if model == "ic" else {"lt_weight": w}
    a = fn(G, seeds, T, 5, edge_checks=True, level_counts_len=12, word_bits=64 * words, graph=captured)
    b = oracle.simulate_threads(model, g, seeds, T, 5, level_counts_len=12, **kw)
    assert np.array_equal(a.spread, b.spread) and np.array_equal(a.node_count, b.node_count)
    assert a.edge_checks == b.edge_checks and np.array_equal(a.level_counts, b.level_counts)
