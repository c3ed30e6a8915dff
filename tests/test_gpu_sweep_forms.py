"""The untuned sweep's forms against a tuned shape that never prefetches, bit for bit: every width and
storage type, a mesh-like graph and its spanning forest (each has its own rule), and blocks that end
just before, on and just after the prefetch distance of 4 MB."""
import numpy as np
import pytest
import torch

from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("K,dt", [(4, torch.float32), (8, torch.float32), (16, torch.float32), (32, torch.float32),
                                  (64, torch.float32), (8, torch.bfloat16), (32, torch.bfloat16),
                                  (64, torch.bfloat16)])
@pytest.mark.parametrize("extra", [-1, 0, 1, 4133])
def test_untuned_form_equals_plain_shape(K, dt, extra):
    import paper_2008_07633_gb300.sfg as S

    n = (4 << 20) // (K * dt.itemsize) + extra
    spec = gen.random_graph(n, 2 * n, seed=K)
    ctx, tuned = S.sfg_ctx_create(0), S.sfg_ctx_create(0)
    for bucket in range(8):
        S.sfg_tune_set(tuned, K, dt, bucket, 3)
    g = S.sfg_laplacian(ctx, n, *(torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in spec[1:]))
    tree, _ = S.sfg_spanning_tree(ctx, g)
    x = torch.from_numpy(gen.gaussian_block(n, K, seed=3)).to(DEV).to(dt)
    for graph in (g, S.sfg_graph_subgraph(ctx, g, tree)):
        outs = [S.sfg_jacobi(c, graph, x.clone(), 3, 0.7) for c in (ctx, tuned)]
        assert torch.equal(*outs)
