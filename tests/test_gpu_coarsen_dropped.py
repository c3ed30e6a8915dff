"""Coarsening a graph that holds edges of infinite weight (parallel edges whose weights add past the FP32 range):
they are left out of the coarse graph and their entry of fine2coarse is -1, like that of an edge inside an
aggregate; backward mapping then skips them."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairs,every", [(2, 1), (50, 7), (40000, 3), (40000, 1000)])
def test_edges_of_infinite_weight(pairs, every):
    import paper_2008_07633_gb300.sfg as S

    # pairs (2i, 2i+1) aggregate; the links (2i+1, 2i+2), every so many of them overflowing
    i = np.arange(pairs - 1)
    inf = i % every == 0
    u = np.concatenate([2 * np.arange(pairs), 2 * i + 1, 2 * i[inf] + 1]).astype(np.int32)
    v = np.concatenate([2 * np.arange(pairs) + 1, 2 * i + 2, 2 * i[inf] + 2]).astype(np.int32)
    w = np.concatenate([np.ones(pairs), np.where(inf, 3e38, 1.0), np.full(inf.sum(), 3e38)]).astype(np.float32)
    ctx = S.sfg_ctx_create(0)
    g = S.sfg_laplacian(ctx, 2 * pairs, *(torch.from_numpy(a).cuda() for a in (u, v, w)))
    X = torch.eye(8, device="cuda")[torch.arange(2 * pairs, device="cuda") // 2 % 8].contiguous()
    agg, f2c, c = S.sfg_coarsen(ctx, g, X)
    assert torch.equal(agg.cpu(), torch.arange(2 * pairs, dtype=torch.int32) // 2)
    eu, ev, _ = (t.cpu().numpy() for t in S.sfg_graph_edges(ctx, g))
    link = eu % 2 == 1
    want = np.full(eu.size, -1, np.int32)
    finite = link.copy()
    finite[link] = ~inf
    want[finite] = np.arange(finite.sum())
    assert c.m == finite.sum() and np.array_equal(f2c.cpu().numpy(), want)
    cu, cv, _ = (t.cpu().numpy() for t in S.sfg_graph_edges(ctx, c))
    assert np.array_equal(cu, i[~inf]) and np.array_equal(cv, i[~inf] + 1)
    back = S.sfg_backward_map(ctx, g, agg, f2c, c, torch.ones(c.m, dtype=torch.uint8, device="cuda"))
    assert np.array_equal(back.cpu().numpy() != 0, ~link | finite)
