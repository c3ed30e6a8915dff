"""Selections whose ids come in no order and are sorted at the end: every number of sorting CTAs at which the form of
the sort changes (16 and 17), partial tiles, ranges smaller than a tile, ids over all 32 bits; and a large one
takes a small multiple of the time that ids in order take (17 times as long where each CTA read the whole
table of digit counts)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ne,k", [(300, 7), (257, 256), (5000, 2049), (70000, 32767), (70000, 32768), (70000, 32769), (65537, 65537),
                                  (100003, 69633),
                                  (1000003, 300001), (3000000, 2500001), (3000000, 3000000)])
@pytest.mark.parametrize("wide", [False, True])
def test_ids_in_no_order(ne, k, wide):
    import paper_2008_07633_gb300.sfg as S

    ctx = S.sfg_ctx_create(0)
    g = torch.Generator(device="cuda").manual_seed(ne + k)
    scores = torch.randperm(ne, generator=g, device="cuda").float()  # distinct up to 2^24
    ids = torch.randperm(ne, generator=g, device="cuda")
    if wide:
        ids = ids * ((2 ** 31 - 1) // ne) + torch.randint(0, (2 ** 31 - 1) // ne, (ne,), generator=g, device="cuda")
    ids = ids.int()
    want = ids[scores >= ne - k].sort().values
    assert torch.equal(S.sfg_select_topk(ctx, scores, ids, k), want)


def test_time_of_a_large_selection():
    import paper_2008_07633_gb300.sfg as S

    ctx = S.sfg_ctx_create(0)
    ne, k = 1 << 22, 1 << 21
    scores = torch.rand(ne, device="cuda")
    best = []
    for ids in (torch.arange(ne, device="cuda").int(), torch.randperm(ne, device="cuda").int()):
        out = torch.empty(k, dtype=torch.int32, device="cuda")
        t = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            S.sfg_select_topk(ctx, scores, ids, k, out=out)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        best.append(min(t))
    print(best)
    assert best[1] <= 5 * best[0], best
