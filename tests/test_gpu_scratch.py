"""Scratch that a context keeps between calls: results do not depend on what earlier calls of other
sizes left in it, on a captured call in between, or on other contexts at work in other threads;
trimming gives it back to the device."""
import threading

import numpy as np
import pytest
import torch

from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
SIZES = (500, 60000, 9000, 61000, 700)


@pytest.fixture(scope="module")
def S():
    import paper_2008_07633_gb300.sfg as S
    return S


def graph(S, ctx, n):
    spec = gen.random_graph(n, 3 * n, seed=n)
    return S.sfg_laplacian(ctx, n, *(torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in spec[1:]))


def fresh(S, n):  # a context of its own keeps nothing from before
    ctx = S.sfg_ctx_create(0)
    mask, _ = S.sfg_sparsify(ctx, graph(S, ctx, n), K=16, steps=4, levels=1)
    return mask.cpu()


def test_sizes_streams_and_threads(S):
    want = {n: fresh(S, n) for n in SIZES}
    bad = []

    def work():
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        ctx = S.sfg_ctx_create(0, streams[0])
        for i in range(4):
            for n in SIZES:
                with torch.cuda.stream(streams[i % 2]):
                    ctx.set_stream(streams[i % 2])
                    mask, _ = S.sfg_sparsify(ctx, graph(S, ctx, n), K=16, steps=4, levels=1)
                    if not torch.equal(mask.cpu(), want[n]):
                        bad.append((i, n))
                streams[i % 2].synchronize()

    threads = [threading.Thread(target=work) for _ in range(3)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not bad


def test_captured_call_between_eager_calls(S):
    stream = torch.cuda.Stream()
    ctx = S.sfg_ctx_create(0, stream)
    with torch.cuda.stream(stream):
        g, small = graph(S, ctx, 61000), graph(S, ctx, 9000)
        want = S.sfg_smooth(ctx, g, 16, 4, 0.7, seed=1).clone()
        other = S.sfg_smooth(ctx, small, 16, 4, 0.7, seed=1).clone()
        out = torch.empty_like(want)
    stream.synchronize()
    replay = torch.cuda.CUDAGraph()
    with torch.cuda.graph(replay, stream=stream, capture_error_mode="relaxed"):
        S.sfg_smooth(ctx, g, 16, 4, 0.7, seed=1, out=out)
    for _ in range(3):
        out.zero_()
        with torch.cuda.stream(stream):
            eager = S.sfg_smooth(ctx, small, 16, 4, 0.7, seed=1)
            replay.replay()
            again = S.sfg_smooth(ctx, g, 16, 4, 0.7, seed=1)
        torch.cuda.synchronize()
        assert torch.equal(out, want) and torch.equal(again, want) and torch.equal(eager, other)


def test_trim_gives_the_kept_blocks_back(S):
    ctx = S.sfg_ctx_create(0)
    g = graph(S, ctx, 400000)
    mask, _ = S.sfg_sparsify(ctx, g, K=64, steps=2)      # two blocks of 102 MB and more
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx.trim()
    assert torch.cuda.mem_get_info()[0] - before >= 2 * 400000 * 64 * 4
    again, _ = S.sfg_sparsify(ctx, g, K=64, steps=2)
    assert torch.equal(again, mask)
