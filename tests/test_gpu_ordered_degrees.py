"""Degrees whose sum depends on its order (weights over many orders of magnitude): bit for bit the sum in column
order, for rows on both sides of every class of the build, in the graph and in a subgraph of it; and a power-law
graph with such weights takes little longer to build than with weights of one order."""
import time

import numpy as np
import pytest
import torch

from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def in_order(rp, val):
    return np.array([np.add.accumulate(val[a:b].astype(np.float64))[-1] if b > a else 0.0 for a, b in zip(rp[:-1], rp[1:])])


@pytest.mark.parametrize("lengths", [(31, 32, 33, 63, 64, 65), (255, 256, 257, 258, 1024, 1025), (4096, 4097, 9000, 16384),
                                     (20000, 300, 40)])
@pytest.mark.parametrize("decades", [15, 4, 2.5])  # sums that always, often and seldom round
@pytest.mark.parametrize("narrow_first", [False, True])
def test_degrees_in_column_order(lengths, narrow_first, decades):
    import paper_2008_07633_gb300.sfg as S

    rng = np.random.default_rng(len(lengths) + lengths[0])
    n = 30000
    u = np.concatenate([np.full(d, 7 * h) for h, d in enumerate(lengths)])
    v = np.concatenate([rng.choice(np.arange(1000, n), d, replace=False) for d in lengths])
    w = 10.0 ** rng.uniform(-decades, decades, u.size)
    if narrow_first:  # a row that may be added in any order beside those that may not
        w[u == 0] = rng.uniform(1, 2, (u == 0).sum())
    ctx = S.sfg_ctx_create(0)
    g = S.sfg_laplacian(ctx, n, dev(u.astype(np.int32)), dev(v.astype(np.int32)), dev(w.astype(np.float32)))
    keep = torch.ones(g.m, dtype=torch.uint8, device="cuda")
    for L in (g, S.sfg_graph_subgraph(ctx, g, keep)):
        rp, _, val, _, deg = (t.cpu().numpy() for t in S.sfg_graph_csr(ctx, L))
        assert np.array_equal(deg.view(np.uint64), in_order(rp, val).view(np.uint64))


def test_wide_weights_cost_little():
    import paper_2008_07633_gb300.sfg as S

    n, u, v, _ = gen.chung_lu(300000, seed=5)
    p = np.random.default_rng(2).permutation(u.size)
    u, v = dev(u[p]), dev(v[p])
    gtor = torch.Generator(device="cuda").manual_seed(1)
    z = torch.randn(u.numel(), generator=gtor, device="cuda")
    ctx = S.sfg_ctx_create(0)
    best = {}
    for sigma in (0.1, 3.0):
        w = torch.exp(sigma * z)
        best[sigma] = 1e9
        for _ in range(15):
            torch.cuda.synchronize()
            t = time.perf_counter()
            S.sfg_laplacian(ctx, n, u, v, w)
            best[sigma] = min(best[sigma], time.perf_counter() - t)
    print(best)
    assert best[3.0] <= 1.35 * best[0.1], best
