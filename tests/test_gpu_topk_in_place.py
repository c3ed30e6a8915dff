"""Selection whose output lies over its own inputs: the same ids as into a list of its own, and the entries
of the inputs outside the output unchanged. Lists of more than one CTA's share, ids in and out of order
(the latter are sorted through a second buffer), ties at the threshold."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("ne,k", [(5, 5), (70000, 1), (70000, 33333), (1000003, 500000), (1000003, 1000003)])
def test_output_over_the_inputs(ne, k, ties, ordered):
    import paper_2008_07633_gb300.sfg as S

    ctx = S.sfg_ctx_create(0)
    g = torch.Generator(device="cuda").manual_seed(ne + k)
    scores = torch.rand(ne, generator=g, device="cuda")
    if ties:
        scores = (scores * 7).floor()
    ids = torch.randperm(2 * ne, generator=g, device="cuda")[:ne].int()
    if ordered:
        ids = ids.sort().values
    want = S.sfg_select_topk(ctx, scores, ids, k).clone()
    for at in {0, (ne - k) // 2, ne - k}:  # over the ids
        buf = ids.clone()
        S.sfg_select_topk(ctx, scores, buf, k, out=buf[at:at + k])
        assert torch.equal(buf[at:at + k], want)
        assert torch.equal(buf[:at], ids[:at]) and torch.equal(buf[at + k:], ids[at + k:])
        buf = scores.clone()               # over the scores
        S.sfg_select_topk(ctx, buf, ids, k, out=buf.view(torch.int32)[at:at + k])
        assert torch.equal(buf.view(torch.int32)[at:at + k], want)
        assert torch.equal(buf[:at], scores[:at]) and torch.equal(buf[at + k:], scores[at + k:])
