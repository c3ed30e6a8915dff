"""sfg_select_topk against a full sort under its strict order (score descending, id ascending), over the
forms of its selection: lists of one candidate to some millions (one CTA to all of them), ids in
ascending order and not, thresholds that fall among equal scores (the id digits decide), scores
with infinities, both zeros, subnormals and negative numbers, k at both ends."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def reference(scores, ids, k):
    b = scores.view(np.uint32)
    image = np.where(b & np.uint32(0x80000000), ~b, b | np.uint32(0x80000000))  # total order of the bits
    order = np.lexsort((ids.astype(np.int64), -image.astype(np.int64)))
    return np.sort(ids[order[:k]])


@pytest.mark.parametrize("ne", [1, 31, 32, 33, 1000, 1025, 8193, 70001, 2500003])
@pytest.mark.parametrize("kind", ["plain", "ties", "equal", "special"])
@pytest.mark.parametrize("order", ["ascending", "random"])
def test_topk_forms(ne, kind, order):
    import paper_2008_07633_gb300.sfg as S

    rng = np.random.default_rng(ne)
    scores = np.exp(3 * rng.standard_normal(ne)).astype(np.float32)
    if kind == "ties":
        scores = rng.integers(0, 5, ne).astype(np.float32)
    elif kind == "equal":
        scores[:] = 1.5
    elif kind == "special":
        scores *= rng.choice(np.array([1, -1], np.float32), ne)
        for step, x in ((7, np.inf), (11, -np.inf), (13, 0.0), (17, -0.0), (19, 1e-42), (23, np.finfo(np.float32).min)):
            scores[::step] = np.float32(x)
    ids = np.sort(rng.choice(2 ** 31 - 1, ne, replace=False).astype(np.int32)) if ne < 100000 else \
        (np.arange(ne, dtype=np.int64) * 800).astype(np.int32)
    if order == "random":
        ids = rng.permutation(ids)
    ctx = S.sfg_ctx_create(0)
    sd, idd = torch.from_numpy(scores).to(DEV), torch.from_numpy(ids).to(DEV)
    for k in sorted({1, max(1, ne // 40), (ne + 1) // 2, ne}):
        got = S.sfg_select_topk(ctx, sd, idd, k)
        torch.cuda.synchronize()
        assert np.array_equal(got.cpu().numpy(), reference(scores, ids, k)), k
