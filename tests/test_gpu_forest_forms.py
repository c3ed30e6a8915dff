"""The spanning forest over the forms of its row search, against the oracle's Kruskal, edge for edge:
rows at the edges of the classes (ranked once up to 15 entries, eight-lane groups up to 32, a warp up to
256, segments above), integer weights so that most keys tie on the weight, edges that are not allowed
(whole rows among them), and long monotone chains, whose hooks need more than one flattening pass."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def stars(seed):
    hubs = tuple((100 + 37 * i, d) for i, d in enumerate((1, 14, 15, 16, 17, 31, 32, 33, 64, 255, 256, 257, 400)))
    return gen.hub_graph(n=5000, m=9000, seed=seed, hubs=hubs)


def chain(n):
    u = np.arange(n - 1)
    return n, u.astype(np.int32), (u + 1).astype(np.int32), np.linspace(1, 2, n - 1).astype(np.float32)


@pytest.mark.parametrize("spec", ["stars", "ties", "chain", "grid"])
@pytest.mark.parametrize("allowed", [None, 0.5, 0.0])
def test_forest_forms(spec, allowed):
    import paper_2008_07633_gb300.sfg as S

    n, u, v, w = {"stars": lambda: stars(3), "ties": lambda: stars(4), "chain": lambda: chain(30000),
                  "grid": lambda: gen.grid3d(31, seed=5)}[spec]()
    if spec == "ties":
        w = np.floor(w / 4).astype(np.float32) + 1
    ctx = S.sfg_ctx_create(0)
    g = S.sfg_laplacian(ctx, n, *(torch.from_numpy(a).to(DEV) for a in (u, v, w)))
    og = O.canonicalize(n, u, v, w)
    allow = None
    if allowed is not None:
        allow = (np.random.default_rng(7).random(og.m) < allowed).astype(np.uint8)
        allow[(og.u == 137) | (og.v == 137)] = 0   # a row with nothing left
    got, count = S.sfg_spanning_tree(ctx, g, None if allow is None else torch.from_numpy(allow).to(DEV))
    want = O.mst(og, allow)
    assert np.array_equal(got.cpu().numpy(), want)
    assert count == int(want.sum())
