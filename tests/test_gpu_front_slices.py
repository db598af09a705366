"""The per-sequence kernel with a sequence's tokens split into slices over the blocks of a cluster: matches, vouchers and spans
across the borders of slices, counts that 16 bits do not hold, vocabularies beyond shared memory, the protected pool with and
without competition, ragged batches with sequences far shorter than the longest. Fast mode and given scores are decided in
fp32 with one rounding per operation on both sides: every index is the oracle's."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_11288_b200 as ta
from ta_testlib import Gpu, bf16_bits, oracle_patterns, oracle_policy
from test_gpu_steps import _workload

pytestmark = pytest.mark.gpu

PATS = [[4, 5], [6], [7, 8, 9], [1, 2, 3, 4, 5, 6, 7, 8]]


def _check(w, K, fast, preset="THEOREM", **kw):
    pol = oracle_policy(K, preset, fast=fast, W=32, vocab_size=max(32000, int(w.vocab)), **kw)
    gen = torch.Generator(device="cuda").manual_seed(7)
    Kd, Vd = (torch.randn((1, w.Hkv, w.total, w.d), generator=gen, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    score = torch.empty((1, w.Hkv, w.total), dtype=torch.float32, device="cuda").exponential_(generator=gen)
    g = Gpu(w, pol, K, 1)
    try:
        for _ in range(2):  # the second call finds the first one's scratch
            if fast:
                idx, cnt, ko, vo = g.compress(None, Kd, Vd)
            else:
                idx, cnt, ko, vo = g.compress_scores(score, None, Kd, Vd)
        torch.cuda.synchronize()
        assert g.poll() == ta.TA_OK
        _, V_o, u0_o = oracle.sponsor_mask(w.ids, w.cu, oracle_patterns(w), pol)
        for b in range(w.B):
            o, e = int(w.cu[b]), int(w.cu[b + 1])
            for h in range(w.Hkv):
                u = u0_o[o:e] if fast else oracle.utility(pol.alpha, pol.delta, score[0, h, o:e].cpu().numpy(), None, u0_o[o:e])
                io, co = oracle.select(V_o[o:e], u, K, pol.n_sink, pol.n_recent, pol.k_protected)
                assert int(cnt[0, b, h]) == co, f"b{b} h{h}"
                np.testing.assert_array_equal(idx[0, b, h].cpu().numpy(), io, err_msg=f"b{b} h{h}")
                rows = torch.from_numpy(np.asarray(io[:co], np.int64)).cuda() + o
                np.testing.assert_array_equal(bf16_bits(ko[0, b, h, :co]), bf16_bits(Kd[0, h, rows]))
                np.testing.assert_array_equal(bf16_bits(vo[0, b, h, :co]), bf16_bits(Vd[0, h, rows]))
                assert not ko[0, b, h, co:].any() and not vo[0, b, h, co:].any()
    finally:
        g.close()


@pytest.mark.parametrize("fast", [True, False])
@pytest.mark.parametrize("lengths,K", [([1025], 40), ([4096], 1000), ([2049, 0, 1, 500], 64), ([8193] * 3, 16), ([16384] * 5, 300),
                                       ([16385], 64), ([40000, 100, 0, 1, 33000, 39999], 300), ([131072], 4096),
                                       ([100001, 17000, 70], 16), ([262144], 1000), ([20000] * 20, 33), ([33000] * 80, 8)])
def test_lengths_and_budgets(lengths, K, fast):
    _check(_workload(lengths, PATS, spans=[6, 64, 33, 12], seed=len(lengths) + K, Hq=1, Hkv=1, W=32), K, fast)


@pytest.mark.parametrize("n", [3000, 17000, 70000])
@pytest.mark.parametrize("K", [50, 4000])
def test_patterns_everywhere(n, K):
    # a small alphabet: matches end at a large share of the positions, so that every border of slices is crossed by some, and
    # more tokens are sponsored than the protected slots hold
    rng = np.random.default_rng(n + K)
    pats = [list(rng.integers(0, 4, size=int(rng.integers(1, 9)))) for _ in range(9)]
    w = _workload([n, n // 2], pats, [int(rng.integers(1, 65)) for _ in pats], [float(rng.integers(1, 30)) for _ in pats], alphabet=4,
                  seed=n, Hq=1, Hkv=1, W=32)
    _check(w, K, True, age_steps=2)
    _check(w, K, False, "SEC33")


def test_counts_beyond_16_bits():
    w = _workload([200000, 65535, 65536], [[0, 1, 0, 0, 1, 1, 0, 1]], alphabet=2, seed=5, Hq=1, Hkv=1, W=32)
    w.ids[int(w.cu[1]):] = 1  # counts of exactly 2^16 - 1 and 2^16
    _check(w, 64, True)
    _check(w, 64, False)


@pytest.mark.parametrize("lengths", [[3000, 700], [40000, 33000], [140000]])
def test_vocabulary_beyond_shared_memory(lengths):
    _check(_workload(lengths, PATS, alphabet=150001, seed=2, Hq=1, Hkv=1, W=32), 100, True)
    _check(_workload(lengths, PATS, alphabet=150001, seed=2, Hq=1, Hkv=1, W=32), 100, False)


def test_more_budget_than_tokens():
    _check(_workload([17000, 3000, 4096], PATS, seed=4, Hq=1, Hkv=1, W=32), 4096, True)
    _check(_workload([17000, 3000, 4096], PATS, seed=4, Hq=1, Hkv=1, W=32), 4096, False)
