"""Rings whose weights increase along them: the first round hooks all nodes into one chain, which pointer jumping
flattens. The forest leaves out the lightest edge, in either order of the nodes, and takes no longer than that of a
ring with weights in no order (1.75 times as long where every jumping thread wrote to one word)."""
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


def ring(n, order, weights, g):
    u = torch.arange(n, device="cuda", dtype=torch.int32)
    v = (u + 1) % n
    w = torch.arange(1, n + 1, device="cuda").float()  # exact up to 2^24
    if weights == "random":
        w = w[torch.randperm(n, generator=g, device="cuda")].contiguous()
    if order == "random":
        p = torch.randperm(n, generator=g, device="cuda").int()
        u, v = p[u.long()].contiguous(), p[v.long()].contiguous()
    return u, v, w


@pytest.mark.parametrize("n", [3, 8, 9, 64, 513, 4097, 65536, 1000003])
@pytest.mark.parametrize("order", ["along", "random"])
def test_chains(n, order):
    import paper_2008_07633_gb300.sfg as S

    ctx = S.sfg_ctx_create(0)
    g = torch.Generator(device="cuda").manual_seed(n)
    L = S.sfg_laplacian(ctx, n, *ring(n, order, "increasing", g))
    mask, count = S.sfg_spanning_tree(ctx, L)
    assert count == n - 1
    assert torch.equal(mask != 0, S.sfg_graph_edges(ctx, L)[2] != 1.0)


def test_time_of_a_chain():
    import paper_2008_07633_gb300.sfg as S

    ctx = S.sfg_ctx_create(0)
    g = torch.Generator(device="cuda").manual_seed(1)
    best = {}
    for weights in ("random", "increasing"):
        L = S.sfg_laplacian(ctx, 65536, *ring(65536, "along", weights, g))
        t = []
        for _ in range(15):
            torch.cuda.synchronize()
            a = time.perf_counter()
            S.sfg_spanning_tree(ctx, L)
            t.append(time.perf_counter() - a)
        best[weights] = min(t)
    assert best["increasing"] <= 1.2 * best["random"], best
