"""The surrogate's aggregations over in-rows and out-rows of every length around the lane groups, the
short/long boundary and the work-item size, against the fp64 oracle."""
import numpy as np
import pytest

import oracle.surrogate as S
import paper_2404_17059_gb300 as P
from paper_2404_17059_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LENGTHS = [0, 1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 255, 256, 257, 288, 289, 512, 513, 1025]


@pytest.mark.parametrize("reverse", [False, True])
def test_row_lengths(reverse):
    """Long out-rows, or (reverse) long in-rows."""
    n, rng = 1400, np.random.default_rng(12)
    a = np.concatenate([np.full(d, u) for u, d in enumerate(LENGTHS)] + [np.arange(100, n)])
    b = np.concatenate([rng.permutation(n)[:d] for d in LENGTHS] + [rng.integers(0, n, n - 100)])
    g = I.csr_from_edges(n, b if reverse else a, a if reverse else b)
    p = rng.uniform(0.0, 0.02, size=g.m).astype(np.float32)
    G = P.cnd_graph_create(n, g.row_ptr, g.col, p, None)
    params = I.surrogate_init(6)
    sur = P.cnd_sur_create(G, params)
    OG = S.Graph(g, p)
    seeds = [0, 5, 24, 700]
    # both sides round to bf16 at the same points; a stored value may move by one unit in the last
    # place (2^-8), as in the other comparisons with the oracle
    yhat, _ = P.cnd_sur_forward(sur, seeds)
    np.testing.assert_allclose(yhat, S.forward(params.astype(np.float64), OG, seeds)["yhat"], rtol=0, atol=5e-3)
    y = rng.uniform(0, 1, size=n).astype(np.float32)
    _, grad = P.cnd_sur_loss_grad(sur, seeds, y)
    _, rg, _ = S.loss_and_grad(params.astype(np.float64), OG, seeds, y.astype(np.float64))
    o = 0
    for _, shape in S.param_shapes():
        k = int(np.prod(shape))
        assert np.abs(grad[o:o + k] - rg[o:o + k]).max() <= 0.02 * np.abs(rg[o:o + k]).max() + 1e-7
        o += k
    sc = P.cnd_sur_scores(sur, seeds)
    rs, _ = S.screen_scores(params.astype(np.float64), OG, seeds)
    assert np.abs(sc - rs).max() <= 0.02 * np.abs(rs).max() + 1e-7


def _overflowing_hub():
    """Node 0 reaches 300 nodes; feeders of at most four out-edges reach targets of several in-degrees.  Nothing
    reaches node 0 or the feeders."""
    feeders, degs = np.arange(301, 401), [0, 1, 2, 3, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 40]
    src, dst, k = [np.zeros(300, np.int64)], [np.arange(1, 301)], 0
    for i, d in enumerate(degs):
        src.append(feeders[(k + np.arange(d)) % 100])
        dst.append(np.full(d, 401 + i))
        k += d
    n = 401 + len(degs)
    return I.csr_from_edges(n, np.concatenate(src), np.concatenate(dst)), np.arange(301, n)


def _params(**kw):
    d = {name: np.zeros(shape) for name, shape in S.param_shapes()}
    for k, entries in kw.items():
        for at, v in entries.items():
            d[k][at] = v
    return S.pack(d).astype(np.float32)


def test_overflow_of_one_row_stays_with_its_neighbours():
    """Node 0's hidden features overflow to infinity; nodes that it does not reach keep their values."""
    g, clean = _overflowing_hub()
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, np.full(g.m, 0.01, dtype=np.float32), None)
    sur = P.cnd_sur_create(G, _params(Ws1={(0, 2): 2e38}, b1={1: 1.0}, Ws2={(0, 1): 1.0}, Ws3={(0, 0): 1.0}, wo={0: 1.0}))
    yh, _ = P.cnd_sur_forward(sur, [])
    np.testing.assert_allclose(yh[clean], 1 / (1 + np.exp(-1.0)), rtol=0, atol=1e-5)


def test_overflow_of_one_gradient_row_stays_with_its_neighbours():
    """The same for the transpose: node 0's row of W_n^T e overflows, and nobody has an edge to node 0."""
    g, _ = _overflowing_hub()
    G = P.cnd_graph_create(g.n, g.row_ptr, g.col, np.full(g.m, 0.01, dtype=np.float32), None)
    scores = []
    for big in (0.0, -1e6):
        # unit 2 is positive at the hub only, and carries a head weight near the largest float; unit 5 of the layer
        # below is active everywhere, so that what reaches it counts
        sur = P.cnd_sur_create(G, _params(Ws1={(2, 2): 1.0}, b1={2: -3.0, 1: 1.0}, Ws2={(2, 2): 1.0, (0, 1): 1.0}, b2={5: 1.0},
                                          Ws3={(1, 2): 1.2e-38, (0, 0): 1.0}, Wn3={(1, 5): big, (0, 0): 0.5},
                                          wo={0: 0.5, 1: 3e38}, bo={0: -9.0}))
        scores.append(P.cnd_sur_scores(sur, []))
    assert np.all(np.isfinite(scores[0])) and np.array_equal(scores[0], scores[1])
