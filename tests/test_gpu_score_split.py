"""CTAs per unit of the score kernel: where the rule has to choose between whole units and units spread over a cluster, it
takes the size that was measured to be the fastest on 148 SMs, and the scores are those of one CTA per unit."""
import numpy as np
import pytest
import torch

import paper_2604_11288_b200 as ta
from ta_testlib import SCORE_ATOL, SCORE_RTOL

pytestmark = pytest.mark.gpu
GUARD = 1


def _score(L, B, Hkv, n, W, force):
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
        ta.ta_ctx_set_score_cluster(ctx, force)
        u = torch.full((L + GUARD, Hkv, B * n), float("nan"), device="cuda")
        ta.ta_score_weighted(ctx, pol, batch, Hq, Hkv, d, ta.view(q), ta.view(k), None, u,
                             torch.cuda.current_stream().cuda_stream)
        assert ta.ta_ctx_poll(ctx) == ta.TA_OK
        assert torch.isnan(u[L:]).all(), "wrote behind its output"
        return u[:L].cpu().numpy(), ta.ta_ctx_last_launch_info(ctx)[0]
    finally:
        ta.ta_ctx_destroy(ctx)


@pytest.mark.parametrize("L,B,Hkv,n,W,want", [
    # 256 score rows
    (19, 1, 8, 2048, 64, 2), (24, 1, 8, 2048, 64, 2), (19, 1, 8, 4096, 64, 4), (10, 1, 8, 4096, 64, 4),
    (40, 1, 8, 3000, 64, 2), (8, 1, 8, 1024, 64, 2), (32, 1, 8, 4096, 64, 1),
    # 128 score rows
    (40, 1, 8, 4096, 32, 2), (10, 1, 8, 5000, 32, 4), (19, 1, 8, 5000, 32, 4), (16, 1, 8, 4096, 32, 1)])
def test_fastest_size_is_taken(L, B, Hkv, n, W, want):
    got, size = _score(L, B, Hkv, n, W, 0)
    assert size == want
    ref, one = _score(L, B, Hkv, n, W, 1)
    assert one == 1
    np.testing.assert_allclose(got, ref, rtol=SCORE_RTOL, atol=SCORE_ATOL)


@pytest.mark.parametrize("L,Hkv,n", [(1, 1, 16384), (1, 2, 9001), (1, 4, 6000), (1, 4, 4096), (2, 2, 3700),
                                     (1, 3, 3200)])
def test_more_than_eight_ctas_for_a_handful_of_units(L, Hkv, n):
    # sizes that cannot be asked for: the rule takes them when all units fit at once and a round of jobs is saved (9 CTAs for
    # 25 tiles, 10 for 29, 11 for 32, 12 for 71, 16 for 47 and 128)
    got, size = _score(L, 1, Hkv, n, 32, 0)
    assert 8 < size <= 16
    ref, _ = _score(L, 1, Hkv, n, 32, 1)
    np.testing.assert_allclose(got, ref, rtol=SCORE_RTOL, atol=SCORE_ATOL)


@pytest.mark.parametrize("L,Hkv,n", [(1, 1, 16384), (1, 2, 9001), (1, 4, 6000), (7, 1, 4090)])
def test_more_than_eight_ctas_with_256_rows(L, Hkv, n):
    got, size = _score(L, 1, Hkv, n, 64, 0)
    assert 8 < size <= 16
    ref, _ = _score(L, 1, Hkv, n, 64, 1)
    np.testing.assert_allclose(got, ref, rtol=SCORE_RTOL, atol=SCORE_ATOL)


@pytest.mark.parametrize("n", [1000, 4096])
def test_128_rows_are_as_precise_as_fp32_sums(n):
    # Every term carries the rounding of its exponent (|x| < 32: 2^-20 absolute, 0.7 of it relative) and of its exponential
    # (2^-22), each term's own; the row's normaliser moves all of a row's terms by its own error (2^-22). Over 128 rows the
    # terms' errors average out: 2-norm error at most 2^-20 * 0.7 / sqrt(128) + 2^-22 < 3e-7. (A cubic in 2 of 16: 1.9e-6.)
    L, Hkv, W, d = 2, 4, 32, 128
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    q = torch.randn((L, 1, 4 * Hkv, W, d), generator=g, dtype=torch.bfloat16, device="cuda")
    k = torch.randn((L, 1, Hkv, n, d), generator=g, dtype=torch.bfloat16, device="cuda")
    pol = ta.ta_policy_default(ta.TA_PRESET_THEOREM, 4)
    batch = ta.make_batch(L, 1, n, n, n)
    ctx = ta.ta_ctx_create(0, ta.ta_scratch_bytes(batch, 4 * Hkv, Hkv, d, 4, pol))
    try:
        u = torch.empty((L, Hkv, n), device="cuda")
        ta.ta_score_weighted(ctx, pol, batch, 4 * Hkv, Hkv, d, ta.view(q), ta.view(k), None, u,
                             torch.cuda.current_stream().cuda_stream)
        assert ta.ta_ctx_poll(ctx) == ta.TA_OK
    finally:
        ta.ta_ctx_destroy(ctx)
    t = torch.arange(W - 1, -1, -1, device="cuda", dtype=torch.double)
    w = (pol.alpha + pol.delta * (1 - pol.pension_rho) * pol.pension_rho ** t).view(-1, 1)
    s = torch.einsum("lghd,lgnd->lghn", q.double().view(L, Hkv, 4 * W, d), k[:, 0].double()) / d ** 0.5
    hidden = torch.arange(n, device="cuda").view(1, -1) > torch.arange(n - W, n, device="cuda").view(-1, 1)
    want = (torch.softmax(s.view(L, Hkv, 4, W, n).masked_fill(hidden, float("-inf")), -1) * w).sum((2, 3))
    assert (u.double() - want).norm() / want.norm() < 3e-7


def _weighted(q, k, W):
    """ta_score_weighted of one unit with 128 rows (4 heads, W = 32)."""
    n = k.shape[0]
    pol = ta.ta_policy_default(ta.TA_PRESET_THEOREM, 4)
    batch = ta.make_batch(1, 1, n, n, n)
    ctx = ta.ta_ctx_create(0, ta.ta_scratch_bytes(batch, 4, 1, 128, 4, pol))
    try:
        u = torch.empty((1, 1, n), device="cuda")
        ta.ta_score_weighted(ctx, pol, batch, 4, 1, 128, ta.view(q.view(1, 1, 4, W, 128)), ta.view(k.view(1, 1, 1, n, 128)),
                             None, u, torch.cuda.current_stream().cuda_stream)
        assert ta.ta_ctx_poll(ctx) == ta.TA_OK
    finally:
        ta.ta_ctx_destroy(ctx)
    return u.view(n)


def test_keys_far_below_the_largest_score_zero():
    # Key 5 is 20 * 20 * 128 / sqrt(128) = 4525 above every other key in all rows: their exponentials are 0 in fp32, whichever
    # row and unit computes them. Key 5 takes all of every row: the sum of the rows' weights.
    n, W = 700, 32
    q = torch.full((4 * W, 128), 20.0, dtype=torch.bfloat16, device="cuda")
    k = torch.zeros((n, 128), dtype=torch.bfloat16, device="cuda")
    k[5] = 20.0
    u = _weighted(q, k, W)
    assert u[5] > 0 and torch.isfinite(u).all()
    u[5] = 0
    assert (u == 0).all()


@pytest.mark.parametrize("row", [0, 13, 14, 15, 31])
def test_a_query_that_is_no_number_shows_in_the_keys_it_sees(row):
    n, W = 700, 32
    g = torch.Generator(device="cuda")
    g.manual_seed(row)
    q = torch.randn((4 * W, 128), generator=g, dtype=torch.bfloat16, device="cuda")
    k = torch.randn((n, 128), generator=g, dtype=torch.bfloat16, device="cuda")
    q[row] = float("nan")
    u = _weighted(q, k, W)
    assert torch.isnan(u[:n - W + row + 1]).all()
    assert torch.isfinite(u[n - W + row + 1:]).all()
