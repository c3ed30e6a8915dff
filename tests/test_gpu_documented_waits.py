"""Entry points documented to synchronise: the stream is idle when they return, so their results can be used
from another stream or context without further ordering. Large meshes, whose last kernels take far longer than
the return; graphs with and without hub rows."""
import numpy as np
import pytest
import torch

from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.fixture(scope="module")
def S():
    import paper_2008_07633_gb300.sfg as S
    return S


def edges(hub):
    n, u, v, w = gen.grid3d(100, seed=3)
    if hub:  # one node joined to 1,000 others
        far = np.arange(5000, 505000, 500, dtype=np.int32)
        u, v = np.concatenate([u, np.zeros_like(far)]), np.concatenate([v, far])
        w = np.concatenate([w, np.ones(far.size, np.float32)])
    return n, [torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (u, v, w)]


@pytest.mark.parametrize("hub", [False, True])
def test_the_stream_is_idle_on_return(S, hub):
    n, e = edges(hub)
    stream = torch.cuda.Stream()
    ctx = S.sfg_ctx_create(0, stream)
    torch.cuda.synchronize()
    idle = {}
    with torch.cuda.stream(stream):
        g = S.sfg_laplacian(ctx, n, *e)
        idle["laplacian"] = stream.query()
        tree, _ = S.sfg_spanning_tree(ctx, g)
        idle["spanning_tree"] = stream.query()
        p = S.sfg_graph_subgraph(ctx, g, tree)
        idle["subgraph"] = stream.query()
        X = S.sfg_smooth(ctx, p, 8, 2, seed=1)
        agg, f2c, c = S.sfg_coarsen(ctx, g, X)
        idle["coarsen"] = stream.query()
        ctree, _ = S.sfg_spanning_tree(ctx, c)
        S.sfg_backward_map(ctx, g, agg, f2c, c, ctree)
        idle["backward_map"] = stream.query()
        S.sfg_sparsify(ctx, g, K=8, steps=2, levels=1)
        idle["sparsify"] = stream.query()
        S.sfg_coloring(ctx, g)
        idle["coloring"] = stream.query()
        S.Batch(ctx, [g], K=8, steps=2)
        idle["batch_create"] = stream.query()
    assert all(idle.values()), idle


@pytest.mark.parametrize("hub", [False, True])
def test_graphs_built_on_one_stream_and_used_on_another(S, hub):
    n, e = edges(hub)
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    build, use = S.sfg_ctx_create(0, a), S.sfg_ctx_create(0, b)
    got = []
    for _ in range(3):
        g = S.sfg_laplacian(build, n, *e)
        with torch.cuda.stream(b):
            got.append([t.clone() for t in S.sfg_graph_csr(use, g)] + [S.sfg_smooth(use, g, 16, 3, seed=2)])
        b.synchronize()
    a.synchronize()
    with torch.cuda.stream(b):
        want = [t.clone() for t in S.sfg_graph_csr(use, g)] + [S.sfg_smooth(use, g, 16, 3, seed=2)]
    b.synchronize()
    for row in got:
        assert all(torch.equal(x, y) for x, y in zip(row, want))
