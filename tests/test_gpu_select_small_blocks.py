"""Many short units with a small budget are selected by blocks of 128 or 256 threads: the same result, bit for bit, as the same
layers give a few at a time (blocks of 1024 threads), at the edges of the instances' lengths and budgets, for uniform and ragged
batches with empty and one-token sequences, and nothing behind the outputs."""
import numpy as np
import pytest
import torch

import paper_2604_11288_b200 as ta

pytestmark = pytest.mark.gpu
D, HKV, GUARD = 128, 4, 1


def _run(ctx, pats, pol, lengths, K, ids, score, k, v):
    L, B, total = score.shape[0], len(lengths), sum(lengths)
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lengths)]), dtype=torch.int32, device="cuda")
    batch = ta.make_batch(L, B, 0, max(lengths), total, cu)
    ko = torch.full((L + GUARD, B, HKV, K, D), 7.0, dtype=torch.bfloat16, device="cuda")
    vo = torch.full_like(ko, 7.0)
    idx = torch.full((L + GUARD, B, HKV, K), -7, dtype=torch.int32, device="cuda")
    cnt = torch.full((L + GUARD, B, HKV), -7, dtype=torch.int32, device="cuda")
    ta.ta_compress_scores(ctx, pats, pol, batch, HKV, D, K, ids, score, None, ta.view(k, True), ta.view(v, True), 0, ko, vo, idx, cnt,
                          torch.cuda.current_stream().cuda_stream)
    assert ta.ta_ctx_poll(ctx) == ta.TA_OK
    for x, fill in ((ko, 7.0), (vo, 7.0), (idx, -7), (cnt, -7)):
        assert (x[L:] == fill).all(), "wrote behind its outputs"
    return [x[:L] for x in (idx, cnt, ko.view(torch.int16), vo.view(torch.int16))]


@pytest.mark.parametrize("lengths,K", [([2048] * 10, 64), ([4096, 1, 0, 17, 4095, 2049, 300, 64, 128, 1000], 64), ([4096] * 10, 16),
                                       ([4096, 1, 0, 17, 4095, 2049, 300, 64, 128, 1000], 65), ([4000] * 10, 193),
                                       ([700] * 10, 1), ([4097, 0, 1, 5000] + [900] * 6, 100), ([8192, 3] + [129] * 8, 128), ([8192, 3] + [129] * 8, 129),
                                       ([1000] * 10, 129), ([300] * 3, 64), ([4000, 31, 2000], 40)])
def test_small_blocks_match_large_ones(lengths, K):
    L = 20 if len(lengths) == 10 else 14
    total = sum(lengths)
    g = torch.Generator(device="cuda")
    g.manual_seed(total + K)
    ids = torch.randint(0, 500, (total,), generator=g, dtype=torch.int32, device="cuda")
    score = torch.empty((L, HKV, total), device="cuda").exponential_(generator=g)
    score[:, 1] = torch.round(score[:, 1])  # ties
    k = torch.randn((L, HKV, total, D), generator=g, dtype=torch.bfloat16, device="cuda")
    v = torch.randn((L, HKV, total, D), generator=g, dtype=torch.bfloat16, device="cuda")
    pol = ta.ta_policy_default(ta.TA_PRESET_SEC33, K)
    pol.vocab_size = 500
    sizing = ta.make_batch(L, len(lengths), 0, max(lengths), total, torch.zeros(len(lengths) + 1, dtype=torch.int32, device="cuda"))
    ctx = ta.ta_ctx_create(0, ta.ta_scratch_bytes(sizing, HKV, HKV, D, K, pol))
    pats = ta.ta_patterns_create(ctx, [[5], [6, 7]])
    try:
        all_layers = _run(ctx, pats, pol, lengths, K, ids, score, k, v)
        for l in range(0, L, 3):
            one = _run(ctx, pats, pol, lengths, K, ids, score[l:l + 1].contiguous(), k[l:l + 1], v[l:l + 1])
            for a, b in zip(all_layers, one):
                assert torch.equal(a[l:l + 1], b)
    finally:
        ta.ta_patterns_destroy(pats)
        ta.ta_ctx_destroy(ctx)
