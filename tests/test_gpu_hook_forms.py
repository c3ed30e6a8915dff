"""Aggregation (sfg_coarsen) on graphs whose rows need every form of the neighbour search: short rows,
rows of exactly 256 and 257 entries (the last one left to an eight-lane group and the first one taken
by a CTA), hubs, and distances that tie (equal rows: the smaller id wins) — against the oracle's
aggregation of the same distances, bit for bit."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("K", [4, 32])
def test_hooks(K, ties):
    import paper_2008_07633_gb300.sfg as S

    n, u, v, w = gen.hub_graph()
    X = gen.gaussian_block(n, K, seed=K)
    if ties:
        X = X[np.arange(n) % 3].copy()  # three distinct rows: most distances are equal
    ctx = S.sfg_ctx_create(0)
    g = S.sfg_laplacian(ctx, n, *(torch.from_numpy(a).to(DEV) for a in (u, v, w)))
    og = O.canonicalize(n, u, v, w)
    agg, f2c, coarse = S.sfg_coarsen(ctx, g, torch.from_numpy(X).to(DEV))
    oagg, onc = O.aggregate(og, O.affinity(og, X.astype(np.float64)))
    assert coarse.n == onc
    assert np.array_equal(agg.cpu().numpy(), oagg)
