"""Streams that own a part of the SMs (green contexts): the calls whose CTAs wait for one another fit their
launches to it and give the same bits as on the whole device."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def partial_stream(sms):
    """A stream on about `sms` SMs, made through the CUDA driver API."""
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")

    def call(name, *args):
        st = getattr(cu, name)(*args)
        if st != 0:
            pytest.skip(f"{name}: {st}")

    whole, part, rest = (ctypes.create_string_buffer(4096) for _ in range(3))
    dev, groups, desc, green, stream = ctypes.c_int(), ctypes.c_uint(1), *(ctypes.c_void_p() for _ in range(3))
    call("cuDeviceGet", ctypes.byref(dev), 0)
    call("cuDeviceGetDevResource", dev, whole, 1)  # the SMs
    call("cuDevSmResourceSplitByCount", part, ctypes.byref(groups), whole, rest, 0, sms)
    call("cuDevResourceGenerateDesc", ctypes.byref(desc), part, 1)
    call("cuGreenCtxCreate", ctypes.byref(green), desc, dev, 1)
    call("cuGreenCtxStreamCreate", ctypes.byref(stream), green, 1, 0)
    return torch.cuda.ExternalStream(stream.value)


@pytest.mark.parametrize("side", [40, 110, 700])
def test_results_on_a_part_of_the_device(side):
    import paper_2008_07633_gb300.sfg as S

    stream = partial_stream(16)
    n, u, v, w = gen.grid2d(side, side, seed=2)
    e = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (u, v, w)]
    home, part = S.sfg_ctx_create(0), S.sfg_ctx_create(0)
    out = []
    for ctx in (home, part):
        if ctx is part:
            torch.cuda.synchronize()
            ctx.set_stream(stream)
        g = S.sfg_laplacian(ctx, n, *e)
        mask, count = S.sfg_sparsify(ctx, g, K=16, steps=5, levels=1)
        tree, _ = S.sfg_spanning_tree(ctx, g)
        p, off = S.sfg_graph_subgraph(ctx, g, tree), torch.nonzero(tree == 0).reshape(-1).int()
        torch.cuda.synchronize()
        X = S.sfg_smooth(ctx, g, 16, 5, seed=3)
        scores = S.sfg_filter_score(ctx, g, p, off, 16, 5, seed=3)
        top = S.sfg_select_topk(ctx, scores, off, off.numel() // 3)
        batch = S.Batch(ctx, [g, g], K=16, steps=3).run(7)
        ctx.trim()
        out.append((mask, tree, X, scores, top, batch))
    assert all(torch.equal(a, b) for a, b in zip(*out))
