"""Small graphs, whose embedding runs in one launch, against the oracle on both sides of the sizes where
that path ends (both halves of the grid resident: n * 16-byte vectors a row <= 77,824 lanes for the
filter, twice that for sfg_smooth), with a single step, even and odd step counts, rows longer than
one 8-entry chunk, isolated nodes and both storage types; and replayed from a CUDA graph."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2008_07633_gb300 import inputs as gen
from parity import check_scores, score_condition

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def setup(n, seed):
    import paper_2008_07633_gb300.sfg as S

    spec = gen.random_graph(n - 2, 4 * n, seed=seed)     # the last two nodes are isolated
    ctx = S.sfg_ctx_create(0)
    g = S.sfg_laplacian(ctx, n, *(torch.from_numpy(a).to(DEV) for a in spec[1:]))
    og = O.canonicalize(n, *spec[1:])
    tree, _ = S.sfg_spanning_tree(ctx, g)
    return S, ctx, g, og, tree, S.sfg_graph_subgraph(ctx, g, tree)


@pytest.mark.parametrize("K,n,steps", [(64, 4863, 3), (64, 4865, 4), (32, 9728, 1), (32, 9729, 2), (4, 77824, 5),
                                       (8, 33, 7), (16, 1000, 10), (4, 3, 2)])
def test_small_filter_and_smooth(K, n, steps):
    S, ctx, g, og, tree, p = setup(n, seed=n)
    X = S.sfg_smooth(ctx, g, K, steps, seed=5).cpu().numpy().astype(np.float64)
    ref = O.smooth(og, K, steps, 0.7, 5)
    assert (np.linalg.norm(X - ref, axis=0) <= 1e-5 * np.maximum(np.linalg.norm(ref, axis=0), 1e-300)).all()
    ids = torch.nonzero(tree == 0).reshape(-1).int()
    if ids.numel() == 0:
        return
    scores = S.sfg_filter_score(ctx, g, p, ids, K, steps, seed=5).cpu().numpy()
    keep, idn = tree.cpu().numpy().astype(bool), ids.cpu().numpy()
    XP = O.smooth(O.canonicalize(n, og.u[keep], og.v[keep], og.w[keep]), K, steps, 0.7, 5)
    check_scores(scores, O.score_edges(og, ref, XP, idn), score_condition(og, ref, XP, idn))


@pytest.mark.parametrize("K,storage", [(16, torch.float32), (64, torch.bfloat16)])
def test_small_filter_replays(K, storage):
    S, ctx, g, og, tree, p = setup(1500, seed=3)
    stream = torch.cuda.Stream()
    ids = torch.nonzero(tree == 0).reshape(-1).int()
    eager = S.sfg_filter_score(ctx, g, p, ids, K, 6, seed=9, storage=storage).clone()
    k = ids.numel() // 7
    sel = S.sfg_select_topk(ctx, eager, ids, k).clone()
    out, top = torch.empty_like(eager), torch.empty_like(sel)
    torch.cuda.synchronize()
    ctx.set_stream(stream)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
        S.sfg_filter_score(ctx, g, p, ids, K, 6, seed=9, storage=storage, out=out)
        S.sfg_select_topk(ctx, out, ids, k, out=top)
    for _ in range(3):
        out.zero_()
        top.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, eager) and torch.equal(top, sel)
