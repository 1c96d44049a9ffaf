"""Scores summed over out-rows of every length around the work-item and lane-group boundaries."""
import numpy as np
import pytest

import oracle.surrogate as S
import paper_2404_17059_gb300 as P
from paper_2404_17059_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DEGREES = [0, 1, 7, 8, 9, 31, 32, 33, 255, 256, 257, 511, 512, 513, 3000]


def test_out_scores_over_row_lengths():
    n = 3200
    rng = np.random.default_rng(8)
    src = np.concatenate([np.full(d, u) for u, d in enumerate(DEGREES)])
    dst = np.concatenate([rng.permutation(n)[:d] for d in DEGREES])
    g = I.csr_from_edges(n, src, dst)
    p = rng.uniform(0.01, 1.0, size=g.m).astype(np.float32)
    G = P.cnd_graph_create(n, g.row_ptr, g.col, p, None)
    params = I.surrogate_init(4)
    sur = P.cnd_sur_create(G, params)
    seeds = [3, 40, 2000]
    yhat, _ = P.cnd_sur_forward(sur, seeds)
    q = np.floor(p.astype(np.float64) * 2.0**32).astype(np.float32).astype(np.float64) * 2.0**-32
    y = yhat.astype(np.float64)
    hop = np.zeros(n)
    np.add.at(hop, g.src(), q * (1 - y[g.col]))
    # the same yhat on both sides: only the fp32 sums differ, by at most (terms + 4) * 2^-24 of the
    # sum of the (non-negative) terms
    ref = (1 - y) * (1 + hop)
    np.testing.assert_allclose(P.cnd_sur_onehop(sur, seeds), ref, rtol=(3000 + 4) * 2.0**-24, atol=1e-7)
    # the network's backward rounds e to bf16: 2 % of the largest entry, as for every gradient
    sc = P.cnd_sur_scores(sur, seeds)
    rs, _ = S.screen_scores(params.astype(np.float64), S.Graph(g, p), seeds)
    assert np.abs(sc - rs).max() <= 0.02 * np.abs(rs).max() + 1e-7
