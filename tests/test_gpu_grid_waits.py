"""A grid barrier that runs out (its waits are told to go on until their limit, 20 ms) is reported by every caller: by the call itself where it synchronises, else by the next call that does, once; and the
context stays usable. No entry of a selection that gave up is an unwritten one."""
import numpy as np
import pytest
import torch

from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu
ETIMEOUT = 4


@pytest.fixture()
def at(monkeypatch):
    """A context whose launches of `kernel` run out of their n-th barrier's waits, and a graph."""
    import paper_2008_07633_gb300.sfg as S

    spec = gen.grid2d(60, 50, seed=4)
    edges = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in spec[1:]]

    def make(kernel, n):
        monkeypatch.setenv("SFG_FAULT_GRID_WAIT", f"{kernel}:{n}")
        ctx = S.sfg_ctx_create(0)
        monkeypatch.delenv("SFG_FAULT_GRID_WAIT")
        return S, ctx, S.sfg_laplacian(ctx, spec[0], *edges)

    return make


def expect(S, ctx, g, call):
    with pytest.raises(S.SfgError) as e:
        call()
    assert e.value.status == ETIMEOUT
    ctx.trim()                                                # reported once
    assert int(S.sfg_graph_edges(ctx, g)[0].numel()) == g.m   # and the context works on
    ctx.trim()


@pytest.mark.parametrize("barrier", [1, 2, 3, 4, 5])
def test_spanning_forest(at, barrier):
    S, ctx, g = at("k_mst", barrier)
    expect(S, ctx, g, lambda: S.sfg_spanning_tree(ctx, g))
    expect(S, ctx, g, lambda: S.sfg_sparsify(ctx, g))
    expect(S, ctx, g, lambda: S.Batch(ctx, [g]))


@pytest.mark.parametrize("barrier", [1, 2, 3, 4, 5, 6, 7, 8, 12])  # 12: the last of the id sort
def test_selection(at, barrier):
    S, ctx, g = at("k_topk", barrier)
    ne, k = 100000, 30000
    scores = torch.rand(ne, device="cuda")
    ids = torch.randperm(ne, device="cuda").int()
    out = torch.full((k,), 2 ** 30, dtype=torch.int32, device="cuda")
    S.sfg_select_topk(ctx, scores, ids, k, out=out)           # queued only
    expect(S, ctx, g, ctx.trim)
    assert bool(((out >= -1) & (out < ne)).all())
    if barrier <= 6:                                          # candidates in id order: no sort
        expect(S, ctx, g, lambda: S.sfg_sparsify(ctx, g, K=8, steps=2))
        expect(S, ctx, g, lambda: S.sfg_sparsify(ctx, g, K=8, steps=2, levels=1))


@pytest.mark.parametrize("barrier", [1, 2, 3, 9])
def test_batch_selection(at, barrier):
    S, ctx, g = at("k_topk_seg", barrier)
    plan = S.Batch(ctx, [g, g], K=8, steps=2)
    plan.run(1)
    expect(S, ctx, g, ctx.trim)
    expect(S, ctx, g, lambda: S.sfg_sparsify_batched(ctx, [g, g], K=8, steps=2))


@pytest.mark.parametrize("barrier", [1, 2, 3, 6, 7])
def test_small_graph_embedding(at, barrier):
    S, ctx, g = at("k_small", barrier)
    steps = 5                                                 # 2 + (steps - 1) + 1 barriers, one more to project
    S.sfg_smooth(ctx, g, 8, steps)
    expect(S, ctx, g, ctx.trim)
    if barrier <= 7:
        tree, _ = S.sfg_spanning_tree(ctx, g)
        p, off = S.sfg_graph_subgraph(ctx, g, tree), torch.nonzero(tree == 0).reshape(-1).int()
        S.sfg_filter_score(ctx, g, p, off, 8, steps)
        expect(S, ctx, g, lambda: S.sfg_laplacian(ctx, 2, *(torch.ones(1, dtype=t, device="cuda") * x for t, x in
                                                            ((torch.int32, 0), (torch.int32, 1), (torch.float32, 1)))))
        expect(S, ctx, g, lambda: S.sfg_sparsify(ctx, g, K=8, steps=steps))


def test_without_the_request_nothing_is_reported(at):
    S, ctx, g = at("none", 1)
    mask, count = S.sfg_sparsify(ctx, g)
    ctx.trim()
    assert int(mask.sum()) == count
