"""The column engine (a block per column of trials, state in shared memory) against the oracle and the
pass engine: graph sizes up to the largest that fits, ragged trial counts, rows around the length from
which a whole block expands them, certain and impossible edges, batches of uneven items."""
import numpy as np
import pytest

import oracle
import paper_2404_17059_gb300 as P
from paper_2404_17059_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LC = 40


def _sim(model, G, seeds, T, rng, **kw):
    f = P.cnd_ic_simulate_ex if model == "ic" else P.cnd_lt_simulate_ex
    return f(G, seeds, T, rng, edge_checks=True, level_counts_len=LC, **kw)


def _check(model, g, G, seeds, T, rng, p, w, **kw):
    a = _sim(model, G, seeds, T, rng, **kw)
    okw = {k: kw[k] for k in ("first_trial", "max_levels") if k in kw}
    b = oracle.simulate_threads(model, g, seeds, T, rng, level_counts_len=LC,
                                **({"ic_prob": p} if model == "ic" else {"lt_weight": w}), **okw)
    c = _sim(model, G, seeds, T, rng, word_bits=64, **kw)  # the pass engine
    assert a.status == (P.CND_ELIMIT if b.status == oracle.LIMIT else P.CND_OK) == c.status
    for x in (b, c):
        assert np.array_equal(a.spread, x.spread)
        assert np.array_equal(a.node_count, x.node_count)
        assert a.edge_checks == x.edge_checks
        assert np.array_equal(a.level_counts, x.level_counts)


def _weights(g, seed=1):
    p = I.ic_uniform_random(g, 0.6, graph_seed=seed)
    p[::7] = 0.0
    p[3::11] = 1.0
    return p, I.lt_weighted_cascade(g)


@pytest.mark.parametrize("model", ["ic", "lt"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 1021, 6000, 23_300, 24_400])  # the last does not fit
def test_graph_sizes(model, n):
    rng = np.random.default_rng(n)
    m = 4 * n
    g = I.csr_from_edges(n, rng.integers(0, n, m), rng.integers(0, n, m))  # self-loops, parallel edges
    p, w = _weights(g)
    G = P.cnd_graph_create(n, g.row_ptr, g.col, p, w)
    seeds = rng.integers(0, n, min(n, 9))  # duplicates among them
    _check(model, g, G, seeds, 100, 3, p, w)


@pytest.mark.parametrize("model", ["ic", "lt"])
def test_trial_counts_offsets_and_caps(model):
    g = I.erdos_renyi_m(700, 4200, graph_seed=2)
    p, w = _weights(g)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, p, w)
    seeds = I.uniform_seeds(g.n, 5, 2)
    for T in (1, 3, 4, 5, 31, 32, 33, 63, 65, 1000, 6001):
        _check(model, g, G, seeds, T, (1 << 63) + T, p, w)
    for ft in (64, (1 << 34) - 128):
        _check(model, g, G, seeds, 130, 9, p, w, first_trial=ft)
    for cap in (1, 2, 5):
        _check(model, g, G, seeds, 70, 4, p, w, max_levels=cap)
    for graph in (0, 1):
        _check(model, g, G, [], 70, 4, p, w, graph=graph)


@pytest.mark.parametrize("model", ["ic", "lt"])
def test_long_rows(model):
    # 80 hubs (more than a step sets aside) with rows of 255, 256, 257 and 3,000 edges, all reached at once
    degs = [255, 256, 257, 3000] + [300] * 76
    n = 4000
    rng = np.random.default_rng(6)
    src = np.concatenate([np.full(len(degs), n - 1)] + [np.full(d, u) for u, d in enumerate(degs)])
    dst = np.concatenate([np.arange(len(degs))] + [rng.permutation(n - 1)[:d] for d in degs])
    g = I.csr_from_edges(n, src, dst)
    p, w = _weights(g)
    p[g.src() == n - 1] = 1.0
    G = P.cnd_graph_create(n, g.row_ptr, g.col, p, w)
    _check(model, g, G, [n - 1], 45, 8, p, w)
    _check(model, g, G, list(range(80)), 45, 8, p, w)


def test_many_trials_without_hub_rows():
    g = I.watts_strogatz(9000, 6, 0.05, graph_seed=3)
    p, w = _weights(g)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, p, w)
    seeds = I.uniform_seeds(g.n, 5, 3)
    a = _sim("ic", G, seeds, 20_001, 2)
    b = _sim("ic", G, seeds, 20_001, 2, word_bits=64 * 128)
    assert np.array_equal(a.spread, b.spread) and np.array_equal(a.node_count, b.node_count)
    assert a.edge_checks == b.edge_checks and np.array_equal(a.level_counts, b.level_counts)


@pytest.mark.parametrize("model", ["ic", "lt"])
def test_batches(model):
    g = I.erdos_renyi_m(600, 4000, graph_seed=5)
    p, w = _weights(g)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, p, w)
    f = P.cnd_ic_simulate_batch if model == "ic" else P.cnd_lt_simulate_batch
    for items, trials_of in ((1, (5,)), (40, (0, 1, 64, 100, 7)), (70, (0, 33)), (1100, (3, 0, 40))):
        off, seeds, _, keys = I.batch_items(g.n, items, 1, 6, (1,), graph_seed=items)
        trials = np.array([trials_of[i % len(trials_of)] for i in range(items)], dtype=np.int32)
        a = f(G, off, seeds, trials, keys, node_count=True, edge_checks=True, level_counts_len=LC)
        b = f(G, off, seeds, trials, keys, node_count=True, edge_checks=True, level_counts_len=LC, word_bits=128)
        assert np.array_equal(a.spread, b.spread) and np.array_equal(a.node_count, b.node_count)
        assert a.edge_checks == b.edge_checks and np.array_equal(a.level_counts, b.level_counts)


def test_time_limit_and_bad_device_seed():
    torch = pytest.importorskip("torch")
    g = I.erdos_renyi_m(600, 4000, graph_seed=5)
    p, w = _weights(g)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, p, w)
    with pytest.raises(P.CndError) as ei:
        _sim("ic", G, [1, 2], 4096, 1, timeout_s=1e-9)
    assert ei.value.status == P.CND_ETIMEOUT
    for bad in (-1, g.n):
        with pytest.raises(P.CndError) as ei:
            _sim("ic", G, torch.tensor([1, bad], dtype=torch.int32, device="cuda"), 64, 1)
        assert ei.value.status == P.CND_EINVAL
    _check("ic", g, G, [1, 2], 64, 1, p, w, timeout_s=30.0)


def test_inputs_beyond_the_staging():
    """More than 256 KB of items or seeds: copied from host memory that the call frees before it ends."""
    g = I.erdos_renyi_m(300, 1500, graph_seed=7)
    p, w = _weights(g)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, p, w)
    off, seeds, _, keys = I.batch_items(g.n, 9000, 1, 4, (1,), graph_seed=7)
    trials = np.array([(4, 9, 0, 33)[i % 4] for i in range(9000)], dtype=np.int32)
    a, b = (P.cnd_ic_simulate_batch(G, off, seeds, trials, keys, node_count=True, edge_checks=True, word_bits=wb)
            for wb in (0, 64 * 512))
    assert np.array_equal(a.spread, b.spread) and np.array_equal(a.node_count, b.node_count)
    assert a.edge_checks == b.edge_checks
    many = np.random.default_rng(7).integers(0, 40, 70_000)
    for model in ("ic", "lt"):
        _check(model, g, G, many, 70, 4, p, w)


@pytest.mark.parametrize("model", ["ic", "lt"])
def test_time_limit_ends_a_long_call(model):
    """The columns that are left when the limit passes are not run."""
    import time
    torch = pytest.importorskip("torch")
    g = I.erdos_renyi_m(1000, 10_000, graph_seed=1)
    p, w = I.ic_uniform(g, 0.1), I.lt_weighted_cascade(g)
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, p, w)
    f = P.cnd_ic_simulate_ex if model == "ic" else P.cnd_lt_simulate_ex
    seeds = torch.tensor([1, 2, 3], dtype=torch.int32, device="cuda")

    def seconds(**kw):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        try:
            f(G, seeds, 20_000_000, 1, **kw)
            status = P.CND_OK
        except P.CndError as e:
            status = e.status
        return time.perf_counter() - t0, status

    seconds()
    full, status = seconds()
    assert status == P.CND_OK and full > 0.02
    limited, status = seconds(timeout_s=full / 20)
    assert status == P.CND_ETIMEOUT
    assert limited < full / 5, (limited, full)


@pytest.mark.parametrize("model", ["ic", "lt"])
def test_engine_of_a_call(model):
    """Which of the calls above run in the column engine, and what keeps a call out of it."""
    engine = {}
    for n in (1, 33, 6000, 23_300, 24_400, 30_000):
        rng = np.random.default_rng(n)
        g = I.csr_from_edges(n, rng.integers(0, n, 4 * n), rng.integers(0, n, 4 * n))
        p, w = _weights(g)
        G = P.cnd_graph_create(n, g.row_ptr, g.col, p, w)
        engine[n], bits = P.cnd_sim_plan(G, model, 100)
        assert 4 <= bits <= 32 if engine[n] == "columns" else bits == 128
        if n == 6000:
            for kw in ({"word_bits": 64}, {"chunk_edges": 8}, {"direction": "push"}, {"defer_bits": 2}, {"stats": 2},
                       {"pull_permille": 250}):
                assert P.cnd_sim_plan(G, model, 100, **kw)[0] == "passes"
            for kw in ({"graph": 1}, {"max_levels": 3}, {"first_trial": 64}, {"n_items": 7}):
                assert P.cnd_sim_plan(G, model, 100, **kw)[0] == "columns"
            assert P.cnd_sim_plan(G, model, 0) == ("passes", 0)
            assert P.cnd_sim_plan(G, model, 2**31 - 1, n_items=2**31 - 1)[1] > 0  # no list of the items is made
            with pytest.raises(P.CndError):
                P.cnd_sim_plan(G, model, 100, word_bits=65)
    assert all(engine[n] == "columns" for n in (1, 33, 6000)) and engine[30_000] == "passes"
    assert engine[23_300] == ("columns" if model == "ic" else "passes")
    assert engine[24_400] == "passes"


def test_engine_of_dense_graphs():
    """A column is one block's work: graphs whose edges take one SM longer than the passes' steps stay with those."""
    n, rng = 5000, np.random.default_rng(1)

    def engine(d, p_of, trials, model="ic"):
        g = I.csr_from_edges(n, np.repeat(np.arange(n), d), rng.integers(0, n, n * d))
        G = P.cnd_graph_create(n, g.row_ptr, g.col, p_of(g), I.lt_weighted_cascade(g))
        return P.cnd_sim_plan(G, model, trials)[0]

    for trials in (1, 64, 1000):
        assert engine(200, lambda g: I.ic_uniform(g, 0.05), trials) == "passes"      # branching 10
        assert engine(200, I.ic_weighted_cascade, trials) == "columns"              # branching 1
        assert engine(10, lambda g: I.ic_uniform(g, 0.5), trials) == "columns"      # few edges
        assert engine(400, I.ic_weighted_cascade, trials, "lt") == "passes"
        assert engine(40, I.ic_weighted_cascade, trials, "lt") == "columns"
