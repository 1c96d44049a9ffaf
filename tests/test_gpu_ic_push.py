"""IC push over slots whose pair counts and rows sit at the edges of how lanes hold them: 1 to 33 pairs,
more than a chunk of 32, wide passes with large work items, per-word keys, certain and impossible edges."""
import numpy as np
import pytest

import oracle
import paper_2404_17059_gb300 as P
from paper_2404_17059_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def graph():
    g = I.rmat(11, 14 << 11, graph_seed=9)  # rows from none to several hundred edges
    p = I.ic_uniform_random(g, 0.3, graph_seed=9)
    p[::5] = 0.0
    p[2::9] = 1.0
    return g, p, P.cnd_graph_create(g.n, g.row_ptr, g.col, p, None)


@pytest.mark.parametrize("words", [1, 2, 3, 5, 15, 16, 17, 31, 32, 33, 64, 65, 257, 300])
def test_pair_counts(graph, words):
    g, p, G = graph
    T = 64 * words - 3
    seeds = I.uniform_seeds(g.n, 4, words)  # every seed holds all words
    for kw in ({}, {"chunk_edges": 3}):
        a = P.cnd_ic_simulate_ex(G, seeds, T, 11, edge_checks=True, level_counts_len=16, word_bits=64 * words, **kw)
        b = oracle.simulate_threads("ic", g, seeds, T, 11, ic_prob=p, level_counts_len=16)
        assert np.array_equal(a.spread, b.spread) and np.array_equal(a.node_count, b.node_count)
        assert a.edge_checks == b.edge_checks and np.array_equal(a.level_counts, b.level_counts)


@pytest.mark.parametrize("items,trials", [(3, (64, 130, 1)), (40, (64, 200, 1024)), (50, (640, 0, 3))])
def test_per_word_keys(graph, items, trials):
    g, p, G = graph
    off, seeds, _, keys = I.batch_items(g.n, items, 1, 9, (1,), graph_seed=items)
    tr = np.array([trials[i % 3] for i in range(items)], dtype=np.int32)
    a = P.cnd_ic_simulate_batch(G, off, seeds, tr, keys + np.uint64(1 << 40), node_count=True, edge_checks=True,
                                word_bits=64 * 2048, first_trial=1 << 35)
    checks = 0
    o = 0
    for i in range(items):
        b = oracle.simulate_threads("ic", g, seeds[off[i]:off[i + 1]], int(tr[i]), int(keys[i]) + (1 << 40), ic_prob=p,
                                    first_trial=1 << 35)
        assert np.array_equal(a.spread[o:o + tr[i]], b.spread) and np.array_equal(a.node_count[i], b.node_count)
        checks += b.edge_checks
        o += int(tr[i])
    assert a.edge_checks == checks


def test_wide_work_items():
    """A pass of more than 256 words on a graph large enough for work items of many edges."""
    g = I.barabasi_albert(70_000, 3, graph_seed=2)
    p = I.ic_weighted_cascade(g)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, p, None)
    seeds = I.top_degree_seeds(g, 30)
    T = 64 * 300 - 9
    a = P.cnd_ic_simulate_ex(G, seeds, T, 4, edge_checks=True)
    b = P.cnd_ic_simulate_ex(G, seeds, T, 4, edge_checks=True, word_bits=64 * 64)
    assert np.array_equal(a.spread, b.spread) and np.array_equal(a.node_count, b.node_count)
    assert a.edge_checks == b.edge_checks
    c = oracle.simulate_threads("ic", g, seeds, 100, 4, ic_prob=p)
    assert np.array_equal(a.spread[:100], c.spread)


def test_items_of_wide_passes_follow_the_step():
    """Passes of more than 256 words: a frontier of a few seeds is dealt out edge by edge; on a graph whose steps
    grow past the line of wider items and fall below it again, results stay those of narrow passes."""
    g = I.erdos_renyi_m(70_000, 700_000, graph_seed=2)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, np.zeros(g.m, dtype=np.float32), None)
    seeds = I.top_degree_seeds(g, 6)
    a = P.cnd_ic_simulate_ex(G, seeds, 64 * 300, 1, word_bits=64 * 300, stats=2)
    assert a.stats["passes"] == 1 and a.stats["work_items"] == g.out_degree()[seeds].sum()
    g = I.rmat(14, 16 << 14, graph_seed=2)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, I.ic_uniform(g, 0.1), None)
    seeds, T = I.top_degree_seeds(g, 20), 64 * 1100 - 7
    kw = dict(edge_checks=True, level_counts_len=16)
    b = P.cnd_ic_simulate_ex(G, seeds, T, 3, word_bits=64 * 200, **kw)
    items = {}
    for graph in (0, 1):
        a = P.cnd_ic_simulate_ex(G, seeds, T, 3, word_bits=64 * 1100, graph=graph, stats=2, **kw)
        assert a.stats["passes"] == 1
        items[graph] = a.stats["work_items"]
        assert np.array_equal(a.spread, b.spread) and np.array_equal(a.node_count, b.node_count)
        assert a.edge_checks == b.edge_checks and np.array_equal(a.level_counts, b.level_counts)
    assert items[0] == items[1]
