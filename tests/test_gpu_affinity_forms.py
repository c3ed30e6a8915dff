"""sfg_affinity against its definition in FP64, bit for bit, over the forms of its reads: rows that
can be read by 16-byte vectors and rows that cannot (odd K, a block that is only 4-byte aligned),
and blocks with zeros, subnormals and signed zeros beside normal numbers. sfg_coarsen reads BF16
blocks through the same kernels."""
import numpy as np
import pytest
import torch

from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def definition(u, v, X):
    """delta_e with increasing k, product and sum rounded separately (numpy never fuses them)."""
    X = X.astype(np.float64)
    nn, dot = np.zeros(X.shape[0]), np.zeros(u.size)
    for k in range(X.shape[1]):
        nn = nn + X[:, k] * X[:, k]
        dot = dot + X[u, k] * X[v, k]
    den = nn[u] * nn[v]
    return np.where(den > 0, 1.0 - dot * dot / np.where(den > 0, den, 1.0), 1.0)


@pytest.mark.parametrize("K,offset,special", [(4, 0, False), (32, 0, False), (64, 0, True), (3, 0, True),
                                              (7, 0, False), (8, 1, True), (1, 0, False)])
def test_affinity_bits(K, offset, special):
    import paper_2008_07633_gb300.sfg as S

    n, u, v, w = gen.random_graph(700, 2500, seed=5)
    X = gen.gaussian_block(n, K, seed=K + offset)
    if special:
        X[::5, 0] = 0.0
        X[1::7] = 0.0
        X[2::11, K - 1] = np.float32(1e-42)   # subnormal
        X[3::13] *= np.float32(1e-30)
        X[4::17, K // 2] = np.float32(-0.0)
    ctx = S.sfg_ctx_create(0)
    g = S.sfg_laplacian(ctx, n, *(torch.from_numpy(a).to(DEV) for a in (u, v, w)))
    cu, cv, _ = (t.cpu().numpy() for t in S.sfg_graph_edges(ctx, g))
    flat = torch.zeros(n * K + offset, dtype=torch.float32, device=DEV)
    Xd = flat[offset:].view(n, K)
    Xd.copy_(torch.from_numpy(X))
    want = definition(cu, cv, X)
    for f in (S.sfg_affinity, S.sfg_affinity_noalloc):
        got = f(ctx, g, Xd)
        torch.cuda.synchronize()
        assert np.array_equal(got.cpu().numpy().view(np.int64), want.view(np.int64))
