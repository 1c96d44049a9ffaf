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


@pytest.mark.parametrize("n,words", [(5_000_003, 33), (1_300_001, 2), (300_001, 31), (70_001, 1), (40_007, 257)])
def test_full_counters(n, words):
    """Every node active in every trial: spreads and counts of strips up to their longest, all words full."""
    row_ptr = np.full(n + 1, n - 1, dtype=np.int32)
    row_ptr[0] = 0
    G = P.cnd_graph_create(n, row_ptr, np.arange(1, n, dtype=np.int32), np.ones(n - 1, np.float32), None)
    T = 64 * words - 1
    a = P.cnd_ic_simulate_ex(G, np.zeros(1, np.int32), T, 3, edge_checks=True)
    assert (a.spread == n).all() and (a.node_count == T).all() and a.edge_checks == T * (n - 1)


@pytest.mark.parametrize("model", ["ic", "lt"])
@pytest.mark.parametrize("words", [257, 700, 2047])
def test_wide_passes_with_few_words_per_node(model, words):
    """Many one-word items: a listed node holds anything from one to some hundred words, scattered over the pass."""
    g = I.erdos_renyi_m(1500, 6000, graph_seed=words)
    p, w = I.ic_weighted_cascade(g), I.lt_weighted_cascade(g)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, p, w)
    off, seeds, _, keys = I.batch_items(g.n, words, 1, 12, (1,), graph_seed=words)
    seeds[off[:-1]] = 7  # and one node that is in every item
    trials = np.full(words, 37, dtype=np.int32)
    f = P.cnd_ic_simulate_batch if model == "ic" else P.cnd_lt_simulate_batch
    a, b = (f(G, off, seeds, trials, keys, node_count=True, edge_checks=True, level_counts_len=30, direction="push",
              word_bits=64 * wb) for wb in (words, 100))
    assert np.array_equal(a.spread, b.spread) and np.array_equal(a.node_count, b.node_count)
    assert a.edge_checks == b.edge_checks and np.array_equal(a.level_counts, b.level_counts)
