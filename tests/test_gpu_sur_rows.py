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
