"""One-pass scoring (log-sum-exp supplied) of uniform batches: the tiles of all units are cut into equal shares, one per
CTA, over unit borders. Lengths around a tile, fewer tiles than CTAs, shares that start and end inside units, and shares
that span several short units; both row-block counts; against the two-pass result and with guard layers behind it."""
import numpy as np
import pytest
import torch

import paper_2604_11288_b200 as ta
from ta_testlib import SCORE_ATOL, SCORE_RTOL

pytestmark = pytest.mark.gpu
GUARD = 2


@pytest.mark.parametrize("L,B,Hkv,n", [(1, 1, 1, 1), (1, 1, 2, 127), (2, 1, 2, 128), (1, 2, 2, 129), (3, 1, 8, 1000),
                                       (40, 1, 8, 100), (20, 2, 8, 300), (7, 3, 8, 1300)])
@pytest.mark.parametrize("W", [32, 64])
def test_shares_match_two_pass(L, B, Hkv, n, W):
    Hq, d = 4 * Hkv, 128
    g = torch.Generator(device="cuda")
    g.manual_seed(n + W)
    q = torch.randn((L, B, Hq, W, d), generator=g, dtype=torch.bfloat16, device="cuda")
    k = torch.randn((L, B, Hkv, n, d), generator=g, dtype=torch.bfloat16, device="cuda")
    pol = ta.ta_policy_default(ta.TA_PRESET_THEOREM, 4)
    pol.obs_window = W
    batch = ta.make_batch(L, B, n, n, B * n)
    ctx = ta.ta_ctx_create(0, ta.ta_scratch_bytes(batch, Hq, Hkv, d, 4, pol))
    try:
        pos = torch.arange(n - W, n, device="cuda").view(1, -1, 1)
        lse = torch.zeros((L, B, Hq, W), device="cuda")
        for l in range(L):
            for b in range(B):
                s = torch.bmm(q[l, b].double(), k[l, b].double().repeat_interleave(4, 0).transpose(1, 2)) / np.sqrt(d)
                s = s.masked_fill(torch.arange(n, device="cuda").view(1, 1, -1) > pos, float("-inf"))
                x = torch.logsumexp(s, -1)
                lse[l, b] = torch.where(torch.isinf(x), torch.zeros_like(x), x).float()
        two = torch.full((L, Hkv, B * n), float("nan"), device="cuda")
        one = torch.full((L + GUARD, Hkv, B * n), float("nan"), device="cuda")
        st = torch.cuda.current_stream().cuda_stream
        ta.ta_score_weighted(ctx, pol, batch, Hq, Hkv, d, ta.view(q), ta.view(k), None, two, st)
        ta.ta_score_weighted(ctx, pol, batch, Hq, Hkv, d, ta.view(q), ta.view(k), lse, one, st)
        assert ta.ta_ctx_poll(ctx) == ta.TA_OK
        assert torch.isnan(one[L:]).all(), "wrote behind its output"
        np.testing.assert_allclose(one[:L].cpu().numpy(), two.cpu().numpy(), rtol=SCORE_RTOL, atol=SCORE_ATOL)
    finally:
        ta.ta_ctx_destroy(ctx)
