"""Selection of few tokens from long units (the instances that bound the threshold by the threads' largest keys) against a plain
sort: ties across the edge of the budget, one value only, the largest values all in a few threads' hands, as many wanted as the
instance allows and one more, units in one block's registers at 512 and at 1024 threads."""
import numpy as np
import pytest
import torch

import paper_2604_11288_b200 as ta

pytestmark = pytest.mark.gpu
D = 128


@pytest.mark.parametrize("units", [8, 160])  # 1024 threads with 8 keys each; 512 threads, or 1024 beyond 16384 tokens
@pytest.mark.parametrize("n,K", [(4097, 1), (8192, 256), (8000, 257), (8192, 512), (16384, 255), (16001, 64), (20000, 512), (700, 300)])
@pytest.mark.parametrize("kind", ["random", "ties", "constant", "clustered"])
def test_few_wanted_match_a_sort(units, n, K, kind):
    L, Hkv = units // 8, 8
    rng = np.random.default_rng(n + K)
    x = rng.exponential(size=(L, Hkv, n)).astype(np.float32)
    if kind == "ties":
        x = np.floor(x * 4)
    elif kind == "constant":
        x[:] = 1.25
    elif kind == "clustered":  # positions that fall to the same few threads
        x[:, :, 5::512] += 50.0
    pol = ta.ta_policy_default(ta.TA_PRESET_THEOREM, K)
    pol.n_sink = pol.n_recent = pol.k_protected = 0
    pol.alpha, pol.beta, pol.gamma, pol.delta, pol.lambda_ = 1.0, 0.0, 0.0, 0.0, 0.0
    pol.vocab_size = 10
    batch = ta.make_batch(L, 1, n, n, n)
    ctx = ta.ta_ctx_create(0, ta.ta_scratch_bytes(batch, Hkv, Hkv, D, K, pol))
    pats = ta.ta_patterns_create(ctx, [])
    try:
        ids = torch.zeros(n, dtype=torch.int32, device="cuda")
        kv = torch.arange(n, device="cuda", dtype=torch.int32).view(torch.bfloat16).view(n, 2).repeat(1, D // 2)
        kv = kv.view(1, 1, 1, n, D).expand(L, 1, Hkv, n, D).contiguous() if units == 8 else None
        if kv is None:
            kv = torch.arange(n, device="cuda", dtype=torch.int32).view(torch.bfloat16).view(n, 2).repeat(1, D // 2)
            kv = kv.view(1, 1, 1, n, D).expand(1, 1, Hkv, n, D).contiguous()
        view = ta.view(kv)
        if units != 8:
            view.stride_l = 0  # every layer the same rows
        ko = torch.empty((L, 1, Hkv, K, D), dtype=torch.bfloat16, device="cuda")
        vo = torch.empty_like(ko)
        idx = torch.full((L, 1, Hkv, K), -7, dtype=torch.int32, device="cuda")
        cnt = torch.full((L, 1, Hkv), -7, dtype=torch.int32, device="cuda")
        ta.ta_compress_scores(ctx, pats, pol, batch, Hkv, D, K, ids, torch.from_numpy(x).cuda(), None, view, view, 0, ko, vo, idx, cnt,
                              torch.cuda.current_stream().cuda_stream)
        assert ta.ta_ctx_poll(ctx) == ta.TA_OK
        got = idx.cpu().numpy().reshape(L * Hkv, K)
        flat = x.reshape(L * Hkv, n)
        want = np.sort(np.argsort(-flat, axis=1, kind="stable")[:, :K], axis=1)
        np.testing.assert_array_equal(got, want)
        rows = ko.view(torch.int16).view(L * Hkv, K, D)[:, :, :2].contiguous().view(torch.int32)[:, :, 0].cpu().numpy()
        np.testing.assert_array_equal(rows, want)
    finally:
        ta.ta_patterns_destroy(pats)
        ta.ta_ctx_destroy(ctx)
