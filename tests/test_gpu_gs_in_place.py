"""Gauss-Seidel smoothing works in the caller's block: its first call on a graph maps no second one."""
import numpy as np
import pytest
import torch

from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,storage", [(64, torch.float32), (64, torch.bfloat16)])
def test_first_call_needs_no_block_of_its_own(K, storage):
    import paper_2008_07633_gb300.sfg as S

    n, u, v, w = gen.grid2d(900, 900, seed=1)
    ctx = S.sfg_ctx_create(0)
    g = S.sfg_laplacian(ctx, n, *(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (u, v, w)))
    S.sfg_coloring(ctx, g)
    out = torch.empty((n, K), dtype=storage, device="cuda")
    ctx.trim()
    before = torch.cuda.mem_get_info()[0]
    S.sfg_smooth_gs(ctx, g, K, 2, seed=1, storage=storage, out=out)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] < out.numel() * out.element_size()
    assert bool(torch.isfinite(out).all())
