"""The LT pull step (counting form) against the oracle and the push step: in-rows around the lengths at
which they change hands or are split, zero-weight in-edges, pass widths around the words a segment owns,
seeds and saturated targets, several passes, the CUDA-graph loop, batches and level caps."""
import numpy as np
import pytest

import oracle
import paper_2404_17059_gb300 as P
from paper_2404_17059_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LC = 24
IN_DEGREES = [1, 2, 7, 8, 9, 63, 64, 65, 96, 254, 255, 256, 257, 300, 510, 511, 766, 1500]


def _targets():
    """One target per in-degree, fed by 1,600 sources that the seeds reach over chains of two steps; some
    in-edges of weight zero; the targets feed each other and back into the sources."""
    n_src, rng = 1600, np.random.default_rng(3)
    k = len(IN_DEGREES)
    n = n_src + k
    src, dst = [], []
    for i, d in enumerate(IN_DEGREES):
        src.append(rng.permutation(n_src)[:d])
        dst.append(np.full(d, n_src + i))
    for _ in range(3):  # sources among themselves
        src.append(rng.permutation(n_src))
        dst.append(rng.permutation(n_src))
    src.append(np.repeat(np.arange(n_src, n), 40))  # targets back into sources and each other
    dst.append(rng.integers(0, n, 40 * k))
    g = I.csr_from_edges(n, np.concatenate(src), np.concatenate(dst))
    w = I.lt_weighted_cascade(g).copy()
    w[rng.random(g.m) < 0.05] = 0  # the others of a node stay equal
    return g, w


@pytest.fixture(scope="module")
def graph():
    g, w = _targets()
    return g, w, P.cnd_graph_create(g.n, g.row_ptr, g.col, None, w)


def _run(G, seeds, T, rng, **kw):
    return P.cnd_lt_simulate_ex(G, seeds, T, rng, edge_checks=True, level_counts_len=LC, stats=2, **kw)


def _same(a, b):
    assert np.array_equal(a.spread, b.spread)
    assert np.array_equal(a.node_count, b.node_count)
    assert a.edge_checks == b.edge_checks
    assert np.array_equal(a.level_counts, b.level_counts)


@pytest.mark.parametrize("words", [1, 2, 15, 16, 17, 31, 32, 33, 65])
def test_pull_widths_match_oracle(graph, words):
    g, w, G = graph
    T = 64 * words - 5
    seeds = I.uniform_seeds(g.n, 300, words)
    b = oracle.simulate_threads("lt", g, seeds, T, 7, lt_weight=w, level_counts_len=LC)
    pull = _run(G, seeds, T, 7, direction="pull")
    assert pull.stats["pull_steps"] == pull.stats["levels"] > 2 and pull.stats["lt_counters"] == 1
    push = _run(G, seeds, T, 7, direction="push")
    assert push.stats["pull_steps"] == 0
    for a in (pull, push, _run(G, seeds, T, 7), _run(G, seeds, T, 7, direction="pull", graph=1)):
        _same(a, b)
    _same(_run(G, seeds, T, 7, direction="pull", word_bits=64 * ((words + 1) // 2)), b)


def test_pull_caps_offsets_and_seed_sets(graph):
    g, w, G = graph
    for seeds in ([], [0], list(range(1600, g.n)), list(range(0, g.n, 2))):
        for kw in ({}, {"max_levels": 1}, {"max_levels": 3}, {"first_trial": 6400}):
            b = oracle.simulate_threads("lt", g, seeds, 200, 5, lt_weight=w, level_counts_len=LC, **kw)
            _same(_run(G, seeds, 200, 5, direction="pull", **kw), b)


def test_pull_batches(graph):
    g, w, G = graph
    off, seeds, _, keys = I.batch_items(g.n, 37, 1, 200, (1,), graph_seed=2)
    trials = np.array([(64, 0, 130, 1000)[i % 4] for i in range(37)], dtype=np.int32)
    out = [P.cnd_lt_simulate_batch(G, off, seeds, trials, keys, node_count=True, edge_checks=True,
                                   level_counts_len=LC, direction=d, word_bits=wb)
           for d, wb in (("push", 0), ("pull", 0), ("auto", 64 * 40), ("pull", 64 * 7))]
    for a in out[1:]:
        _same(a, out[0])


def test_dense_frontier_pulls_by_itself():
    g = I.rmat(15, 16 << 15, graph_seed=4)
    w = I.lt_weighted_cascade(g)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, None, w)
    seeds = I.top_degree_seeds(g, 100)
    push = _run(G, seeds, 1000, 2, direction="push")
    for graph in (0, 1):
        a = _run(G, seeds, 1000, 2, graph=graph)
        assert 0 < a.stats["pull_steps"] < a.stats["levels"]
        _same(a, push)


@pytest.mark.parametrize("words", [1, 2, 3, 16, 17, 40])
def test_word_checks_of_a_pull_step(words):
    """Every in-edge comes from a seed and no target activates: one pull step, which reads the words of the pass
    once for each in-edge, whatever it pads its lists and lanes with."""
    k = len(IN_DEGREES)
    n = 1600 + k
    g = I.csr_from_edges(n, np.concatenate([np.arange(d) for d in IN_DEGREES]), np.repeat(np.arange(1600, n), IN_DEGREES))
    G = P.cnd_graph_create(n, g.row_ptr, g.col, None, np.ones(g.m, dtype=np.uint32))
    seeds = np.arange(1600)
    a = _run(G, seeds, 64 * words - 5, 1, direction="pull", word_bits=64 * words)
    assert np.all(a.spread == 1600) and a.stats["pull_steps"] == a.stats["levels"] == 1
    assert a.stats["word_checks"] == g.m * words


def test_pass_width_has_room_for_the_frontier_rows():
    """The words of a pass, planned for little free memory: its state, the pull's rows by node among it, stays
    within 60 % of that."""
    g = I.erdos_renyi_m(50_000, 200_000, graph_seed=3)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, I.ic_uniform(g, 0.1), I.lt_weighted_cascade(g))
    planes = sum(int(k).bit_length() for k in g.in_degree())
    free = 100 << 20
    state = 2 * 8 + 2 * 10  # per node and word: vis, nxt, two pools
    for model, kw, per_word in (("lt", {}, g.n * (state + 8) + 8 * planes), ("lt", {"direction": "push"}, g.n * state + 8 * planes),
                                ("ic", {"pull_permille": 250}, g.n * (state + 8)), ("ic", {}, g.n * state)):
        engine, bits = P.cnd_sim_plan(G, model, 10_000_000, free_bytes=free, **kw)
        words = bits // 64
        assert engine == "passes" and words > 8
        assert words * per_word <= 0.6 * free < (words + 4) * per_word, (model, kw, words)


def test_graph_loop_without_pulls_launches_none():
    """The CUDA-graph loop of a sparse cascade runs three kernels a step; from the first step that pulls on, six."""
    for g, pulls in ((I.erdos_renyi_m(30_000, 300_000, graph_seed=4), False), (I.rmat(15, 16 << 15, graph_seed=4), True)):
        w = I.lt_weighted_cascade(g)
        G = P.cnd_graph_create(g.n, g.row_ptr, g.col, None, w)
        seeds = I.top_degree_seeds(g, 100 if pulls else 2)
        push = _run(G, seeds, 1000, 2, direction="push", graph=1)
        a = _run(G, seeds, 1000, 2, graph=1)
        _same(a, push)
        s, base = a.stats, push.stats["launches"] - 3 * push.stats["levels"]  # outside the loop
        assert s["levels"] == push.stats["levels"] and (s["pull_steps"] > 0) == pulls
        extra = s["launches"] - base - 3 * s["levels"]
        assert extra == 0 if not pulls else 3 * s["pull_steps"] <= extra <= 3 * s["levels"]


def test_small_steps_push():
    """Steps of few checks have nothing to save by pulling, however dense their frontier."""
    g = I.erdos_renyi_m(30_000, 120_000, graph_seed=4)
    w = I.lt_weighted_cascade(g)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, None, w)
    seeds = I.top_degree_seeds(g, 3000)
    for T in (64, 400):
        a = _run(G, seeds, T, 2)
        assert a.stats["pull_steps"] == 0
        _same(a, _run(G, seeds, T, 2, direction="pull"))
