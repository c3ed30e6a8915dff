"""Lists with rows of more than 16,384 raw entries, which are sorted apart from the others: bit for bit the graph
(and, through coarsening, the edge map) of the sort of all entries, for one and several such rows, next to
rows at the edge of the class; parallel edges in runs across the eight-entry reads; weights narrow enough for the
parallel degree sum and weights that need the ordered one; hubs among the first and the last columns."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def edges(hubs, lengths, n, dup, wide, order, seed, share):
    rng = np.random.default_rng(seed)
    rest = int(sum(lengths) / (2 * share) - sum(lengths))  # the hub rows hold about `share` of the entries
    u, v = [rng.integers(0, n, rest)], [rng.integers(0, n, rest)]  # self-loops and repeats among them
    for h, d in zip(hubs, lengths):
        u.append(np.full(d, h))
        v.append(rng.integers(0, n // 40, d) if dup else rng.choice(n, d, replace=False))
    u, v = np.concatenate(u), np.concatenate(v)
    flip = rng.random(u.size) < 0.5
    u, v = np.where(flip, v, u), np.where(flip, u, v)
    p = rng.permutation(u.size) if order == "random" else np.lexsort((np.maximum(u, v), np.minimum(u, v)))
    w = 10.0 ** rng.uniform(-12, 12, u.size) if wide else rng.uniform(0.5, 2.0, u.size)
    return [torch.from_numpy(a[p]).cuda() for a in (u.astype(np.int32), v.astype(np.int32), w.astype(np.float32))]


@pytest.mark.parametrize("hubs,lengths,n,share", [((0,), (16400,), 17000, 0.1), ((40000,), (39000,), 40001, 0.2),
                                                  ((5, 20000, 39999), (16384, 16390, 40000), 40000, 0.05),
                                                  (tuple(range(100, 230)), (16500,) * 130, 90000, 0.15),  # several sorts
                                                  ((5, 7), (30000, 20000), 40000, 0.4)])                  # the sort of all
@pytest.mark.parametrize("dup,wide,order", [(False, False, "random"), (True, True, "random"), (True, False, "sorted"),
                                            (False, True, "sorted")])
def test_against_the_sort_of_all_entries(monkeypatch, hubs, lengths, n, share, dup, wide, order):
    import paper_2008_07633_gb300.sfg as S

    e = edges(hubs, lengths, n, dup, wide, order, len(hubs), share)
    rows = S.sfg_ctx_create(0)
    monkeypatch.setenv("SFG_BUILD_SORT", "1")
    sort = S.sfg_ctx_create(0)
    monkeypatch.delenv("SFG_BUILD_SORT")
    X = torch.randn((n, 8), generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    X[:n // 2] = X[:n // 2].abs()                       # near-parallel rows: large aggregates, long coarse rows
    out = []
    for ctx in (rows, sort):
        g = S.sfg_laplacian(ctx, n, *e)
        agg, f2c, c = S.sfg_coarsen(ctx, g, X)
        out.append([*S.sfg_graph_edges(ctx, g), *S.sfg_graph_csr(ctx, g), agg, f2c, *S.sfg_graph_edges(ctx, c),
                    *S.sfg_graph_csr(ctx, c)])
    for a, b in zip(*out):
        assert torch.equal(a, b)
