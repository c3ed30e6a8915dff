"""One hub row does not change how the other rows of a mesh are swept: the tile kernel takes as long as on the mesh
without it (1.25-1.45 times as long where the form went by the presence of a hub row), and the sweeps agree with
the oracle on meshes with hub rows and on graphs whose rows differ widely in length."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def with_hub(n, u, v, w, deg):
    far = np.random.default_rng(1).permutation(n - 1)[:deg].astype(np.int32) + 1
    return n, np.concatenate([u, np.zeros_like(far)]), np.concatenate([v, far]), np.concatenate([w, np.ones(deg, np.float32)])


def tile_kernel_ms(S, ctx, g, K, storage):
    X = torch.randn(g.n, K, device="cuda").to(storage)
    best = 1e9
    for _ in range(6):
        S.sfg_ctx_timing(ctx, True)
        S.sfg_jacobi(ctx, g, X, 12)
        best = min(best, S.sfg_ctx_kernel_time(ctx, "jacobi")[1] - S.sfg_ctx_kernel_time(ctx, "jacobi_heavy")[1])
    S.sfg_ctx_timing(ctx, False)
    return best


@pytest.mark.parametrize("K,storage", [(32, torch.float32), (64, torch.float32), (32, torch.bfloat16)])
def test_a_hub_row_leaves_the_mesh_form(K, storage):
    import paper_2008_07633_gb300.sfg as S

    ctx = S.sfg_ctx_create(0)
    n, u, v, w = gen.grid3d(128, seed=2)
    plain = S.sfg_laplacian(ctx, n, dev(u), dev(v), dev(w))
    hub = S.sfg_laplacian(ctx, n, *(dev(a) for a in with_hub(n, u, v, w, 1000)[1:]))
    assert tile_kernel_ms(S, ctx, hub, K, storage) <= 1.12 * tile_kernel_ms(S, ctx, plain, K, storage)


@pytest.mark.parametrize("spec", [with_hub(*gen.grid2d(70, 60, seed=3), 400), gen.chung_lu(6000, seed=5),
                                  gen.hub_graph(6000, 15000, seed=31)], ids=["mesh", "chung_lu", "hubs"])
@pytest.mark.parametrize("K", [4, 32, 64])
def test_sweeps_against_the_oracle(spec, K):
    import paper_2008_07633_gb300.sfg as S

    n, u, v, w = spec[:4]
    ctx = S.sfg_ctx_create(0)
    g = S.sfg_laplacian(ctx, n, dev(u), dev(v), dev(w))
    X = S.sfg_smooth(ctx, g, K, 5, seed=5).cpu().numpy().astype(np.float64)
    ref = O.smooth(O.canonicalize(n, u, v, w), K, 5, 0.7, 5)
    assert (np.linalg.norm(X - ref, axis=0) <= 1e-5 * np.maximum(np.linalg.norm(ref, axis=0), 1e-300)).all()
