"""The Laplacian build over the forms of its row sort, bit for bit against the oracle: raw rows at
the edges of the three classes (ranked up to 32 entries, one CTA up to 1,024 and up to 16,384) and one
past the last (which sends the whole list through the radix sort); parallel edges and self-loops;
weights narrow enough for the parallel degree sum and weights that need the ordered one; sorted
lists, whose warps share an endpoint."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def star_lists(lengths, dup, wide, order, seed):
    rng = np.random.default_rng(seed)
    n = 40000 + len(lengths)
    u, v = [], []
    for h, d in enumerate(lengths):  # hub ids spread over the range, so hubs have columns on both sides
        hub = h * 97 + 500
        k = min(d // 3, 500)
        if dup:
            leaves, low = rng.integers(len(lengths) * 97 + 600, n, d - k), rng.integers(0, 500, k)
        else:
            leaves, low = rng.choice(np.arange(20000, n), d - k, replace=False), rng.choice(np.arange(500), k, replace=False)
        leaves = np.concatenate([leaves, low])
        flip = rng.random(leaves.size) < 0.5
        u.append(np.where(flip, hub, leaves))
        v.append(np.where(flip, leaves, hub))
    u, v = np.concatenate(u), np.concatenate(v)
    loops = rng.integers(0, n, 9)
    u, v = np.concatenate([u, loops]), np.concatenate([v, loops])
    p = rng.permutation(u.size) if order == "random" else np.lexsort((np.maximum(u, v), np.minimum(u, v)))
    w = 10.0 ** rng.uniform(-12, 12, u.size) if wide else rng.uniform(0.5, 2.0, u.size)
    return n, u[p].astype(np.int32), v[p].astype(np.int32), w.astype(np.float32)


@pytest.mark.parametrize("lengths", [(1, 2, 31, 32, 33, 64), (255, 256, 257, 1023, 1024, 1025, 1500), (4095, 4096, 4097, 33), (5000, 16384, 40), (257, 1024, 1025),
                                     (16385, 33, 8)])
@pytest.mark.parametrize("dup,wide,order", [(False, False, "random"), (True, True, "random"), (True, False, "sorted")])
def test_rows_bit_exact(lengths, dup, wide, order):
    import paper_2008_07633_gb300.sfg as S

    n, u, v, w = star_lists(lengths, dup, wide, order, seed=sum(lengths))
    ctx = S.sfg_ctx_create(0)
    g = S.sfg_laplacian(ctx, n, *(torch.from_numpy(a).to(DEV) for a in (u, v, w)))
    og = O.canonicalize(n, u, v, w)
    cu, cv, cw = (t.cpu().numpy() for t in S.sfg_graph_edges(ctx, g))
    assert np.array_equal(cu, og.u) and np.array_equal(cv, og.v)
    assert np.array_equal(cw.view(np.uint32), og.w.view(np.uint32))
    rp, col, val, eid, deg = (t.cpu().numpy() for t in S.sfg_graph_csr(ctx, g))
    orp, ocol, oval, oeid, odeg = O.laplacian_csr(og)
    assert np.array_equal(rp, orp) and np.array_equal(col, ocol) and np.array_equal(eid, oeid)
    assert np.array_equal(val.astype(np.float64), oval)
    assert np.array_equal(deg.view(np.uint64), odeg.view(np.uint64))
