"""Kept scratch and the life of streams and contexts: a context that moves from a destroyed stream with work
pending to a new one (whose handle may be the old one's), the per-thread default stream used from several
threads, contexts destroyed while their stream is being captured, and an allocation that finds the pool out
of memory while another, idle context keeps scratch."""
import ctypes
import threading

import numpy as np
import pytest
import torch

from paper_2008_07633_gb300 import inputs as gen

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.fixture(scope="module")
def S():
    import paper_2008_07633_gb300.sfg as S
    torch.zeros(1, device=DEV)
    return S


def graph(S, ctx, side):
    n, u, v, w = gen.grid2d(side, side, seed=side)
    return S.sfg_laplacian(ctx, n, *(torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (u, v, w)))


def driver(name, *args):
    st = getattr(ctypes.CDLL("libcuda.so.1"), name)(*args)
    assert st == 0, (name, st)


def new_stream():
    h = ctypes.c_void_p()
    driver("cuStreamCreate", ctypes.byref(h), ctypes.c_uint(1))  # non-blocking
    return torch.cuda.ExternalStream(h.value, device=DEV)


def destroy(stream):
    driver("cuStreamDestroy_v2", ctypes.c_void_p(stream.cuda_stream))


def test_streams_destroyed_with_work_pending(S):
    ctx = S.sfg_ctx_create(0)
    g = graph(S, ctx, 600)
    want = [S.sfg_smooth(ctx, g, 64, 6, seed=i).clone() for i in range(12)]
    got = [torch.empty_like(x) for x in want]
    home = torch.cuda.current_stream()
    torch.cuda.synchronize()
    for i, out in enumerate(got):
        stream = new_stream()
        ctx.set_stream(stream)
        S.sfg_smooth(ctx, g, 64, 6, seed=i, out=out)
        destroy(stream)
    ctx.set_stream(home)
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(got, want))


def test_per_thread_default_stream(S):
    ctx = S.sfg_ctx_create(0)
    g = graph(S, ctx, 500)
    want = [S.sfg_smooth(ctx, g, 32, 6, seed=i).clone() for i in range(8)]
    got = [torch.empty_like(x) for x in want]
    torch.cuda.synchronize()
    home = torch.cuda.current_stream()
    ctx.set_stream(torch.cuda.ExternalStream(2, device=DEV))  # cudaStreamPerThread: one stream a thread
    for i, out in enumerate(got):  # one thread after the other, none waiting for its stream
        t = threading.Thread(target=lambda: S.sfg_smooth(ctx, g, 32, 6, seed=i, out=out))
        t.start()
        t.join()
    torch.cuda.synchronize()
    ctx.set_stream(home)
    assert all(torch.equal(x, y) for x, y in zip(got, want))


def kept(S, stream=None):
    """A context that keeps scratch (an 18 MB and a 92 MB block among others), and a graph of its own."""
    ctx = S.sfg_ctx_create(0, stream)
    g = graph(S, ctx, 600)
    S.sfg_smooth(ctx, g, 64, 2)
    torch.cuda.synchronize()
    return ctx, g


def unused(S, ctx):
    ctx.trim()
    return torch.cuda.mem_get_info()[0]


def test_between_the_legacy_stream_and_others(S):
    home, side = torch.cuda.current_stream(), torch.cuda.Stream()
    ctx = S.sfg_ctx_create(0)
    g = graph(S, ctx, 500)
    want = [S.sfg_smooth(ctx, g, 64, 6, seed=i).clone() for i in range(10)]
    got = [torch.empty_like(x) for x in want]
    torch.cuda.synchronize()
    for i, out in enumerate(got):  # neither stream waits for the other
        ctx.set_stream(side if i % 2 else home)
        S.sfg_smooth(ctx, g, 64, 6, seed=i, out=out)
    ctx.set_stream(home)
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(got, want))


@pytest.mark.parametrize("own_stream", [False, True])
def test_an_allocation_takes_back_what_idle_contexts_keep(S, monkeypatch, own_stream):
    other = S.sfg_ctx_create(0)
    small = graph(S, other, 40)
    idle, g = kept(S, torch.cuda.Stream() if own_stream else None)
    before = unused(S, other)                     # the idle context's blocks stay
    monkeypatch.setenv("SFG_FAULT_POOL", "3")
    ctx = S.sfg_ctx_create(0)
    monkeypatch.delenv("SFG_FAULT_POOL")
    ref, x = S.sfg_smooth(other, small, 8, 3, seed=1), S.sfg_smooth(ctx, small, 8, 3, seed=1)
    assert torch.equal(x, ref)
    assert unused(S, ctx) - before >= 80 << 20    # now they have gone back to the device
    y = S.sfg_smooth(idle, g, 64, 2)              # whose owner works on
    assert torch.equal(y, S.sfg_smooth(other, g, 64, 2))


def test_a_context_destroyed_while_its_stream_is_captured(S):
    other = S.sfg_ctx_create(0)
    graph(S, other, 40)
    stream = new_stream()
    ctx, g = kept(S, stream)
    g.close()
    torch.cuda.synchronize()
    before = unused(S, other)
    driver("cuStreamBeginCapture_v2", ctypes.c_void_p(stream.cuda_stream), ctypes.c_int(2))  # relaxed
    ctx.close()
    graph_h = ctypes.c_void_p()
    driver("cuStreamEndCapture", ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph_h))  # still valid
    driver("cuGraphDestroy", graph_h)
    torch.cuda.synchronize()
    assert unused(S, other) - before >= 80 << 20
    destroy(stream)


def test_repeated_contexts_give_all_their_room_back(S):
    # the share of all contexts is bounded: a context that left with blocks on its account would lower it
    for _ in range(200):
        ctx, g = kept(S)
        g.close()
        ctx.close()
    other = S.sfg_ctx_create(0)
    idle, g = kept(S)
    before = unused(S, other)
    assert unused(S, idle) - before >= 80 << 20   # the last one still kept its blocks


def test_taking_back_beside_contexts_at_work(S, monkeypatch):
    bad, stop = [], threading.Event()
    ref_ctx = S.sfg_ctx_create(0)
    refs = {side: S.sfg_smooth(ref_ctx, graph(S, ref_ctx, side), 32, 4, seed=side).clone() for side in (30, 200, 500)}
    torch.cuda.synchronize()

    def work(own_stream):
        stream = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
        ctx = S.sfg_ctx_create(0, stream)
        with torch.cuda.stream(stream):
            graphs = {side: graph(S, ctx, side) for side in refs}
            while not stop.is_set():
                for side, g in graphs.items():
                    if not torch.equal(S.sfg_smooth(ctx, g, 32, 4, seed=side), refs[side]):
                        bad.append(side)
        stream.synchronize()

    threads = [threading.Thread(target=work, args=(o,)) for o in (False, True, True)]
    [t.start() for t in threads]
    for n in range(1, 40):
        monkeypatch.setenv("SFG_FAULT_POOL", str(n))
        ctx = S.sfg_ctx_create(0)
        g = graph(S, ctx, 200)
        if not torch.equal(S.sfg_smooth(ctx, g, 32, 4, seed=200), refs[200]):
            bad.append(("reclaiming", n))
        g.close()
        ctx.close()
    monkeypatch.delenv("SFG_FAULT_POOL")
    stop.set()
    [t.join() for t in threads]
    assert not bad
