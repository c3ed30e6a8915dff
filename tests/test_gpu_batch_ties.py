"""The batch plan's selection where every score of a graph ties: with no sweep both embeddings are the
same block and every ratio is one, so each graph must take its smallest candidate ids, from lists of
one candidate, around one warp's and one CTA's range, and of tens of thousands."""
import numpy as np
import pytest
import torch

from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("frac", [0.001, 0.05, 0.5])
def test_ties_take_the_smallest_ids(frac):
    import paper_2008_07633_gb300.sfg as S

    ctx = S.sfg_ctx_create(0)
    specs = [gen.random_graph(n, m, seed=i) for i, (n, m) in enumerate(
        [(3, 3), (20, 33), (40, 72), (300, 1290), (1000, 9200), (9000, 90000)])]
    specs.insert(2, gen.path(40, weights="uniform"))  # a tree: no candidate
    gs = [S.sfg_laplacian(ctx, n, *(torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in e))
          for n, *e in specs]
    plan = S.Batch(ctx, gs, K=16, steps=0, budget_frac=frac)
    for g, mask, count in zip(gs, plan.split(plan.run(5)), plan.counts):
        tree, _ = S.sfg_spanning_tree(ctx, g)
        tree = tree.cpu().numpy().astype(bool)
        want = tree.copy()
        want[np.flatnonzero(~tree)[: count - int(tree.sum())]] = True
        assert np.array_equal(mask.cpu().numpy().astype(bool), want)
