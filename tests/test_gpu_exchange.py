"""What the CTAs of a cluster tell one another while they search a unit together (sequences of more than 16384 tokens): candidates
that all lie in one CTA's slice, so that most CTAs have none to send and one has none to receive. Decided in fp32 with one rounding
per operation on both sides: every index is the oracle's."""
import time

import numpy as np
import pytest
import torch

import paper_2604_11288_b200 as ta
from ta_testlib import Gpu, oracle_policy
from test_gpu_front_slices import _check
from test_gpu_steps import _select_case, _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 8, 20, 40])  # 16, 8, 4 and 2 CTAs to a sequence on 148 SMs
@pytest.mark.parametrize("at", [0.0, 0.47, 0.93])
@pytest.mark.parametrize("fast", [True, False])
def test_sponsored_tokens_in_one_slice(batch, at, fast):
    # more of them than protected slots, and fewer than the list of candidates holds: the first exchange after the ranges is theirs;
    # fast mode: recency leaves the main pool's last candidates to the last slice
    w = _workload([20000] + [17000 + 40 * b for b in range(batch - 1)], [[31999], [31998, 31997]], [7, 40], [9.0, 13.0], alphabet=31000,
                  seed=batch, Hq=1, Hkv=1, W=32)
    rng = np.random.default_rng(batch)
    for b in range(w.B):
        o, n = int(w.cu[b]), int(w.lengths[b])
        run = w.ids[o + int(at * n):o + int(at * n) + 600]
        run[rng.integers(0, 598, size=25)] = 31999
        for i in rng.integers(0, 598, size=25):
            run[i:i + 2] = [31998, 31997]
    _check(w, 64, fast, "AUDIT")


@pytest.mark.parametrize("lengths,L", [([20000, 9000, 300], 1), ([100000], 1), ([200000], 2)])  # blocks of 512, 1024, 1024 threads
@pytest.mark.parametrize("at", [0.0, 0.3, 0.96])
def test_candidates_in_one_slice(lengths, L, at):
    # a run of close neighbours far above everything else, the threshold among them
    w = _workload(lengths, [[5, 6, 7], [9]], seed=L, Hq=1, Hkv=1)
    gen = torch.Generator().manual_seed(len(lengths))
    A = torch.rand((L, 1, w.total), generator=gen) / 4
    for b in range(w.B):
        i = int(w.cu[b]) + int(at * int(w.lengths[b]))
        m = min(500, int(w.cu[b + 1]) - i)
        A[:, :, i:i + m] = 64.0 + torch.rand((L, 1, m), generator=gen) / 1024
    _select_case(w, oracle_policy(100, "AUDIT", beta=0.0, gamma=0.0, lam=0.0), 100, L, (A.cuda(), torch.zeros_like(A).cuda()))


@pytest.mark.parametrize("stop", [0, 1, 2, 3, 4])
def test_a_search_whose_peer_stops_taking_part_ends(stop):
    # (the one that stops does so by sending nothing more; both stay until the other is done)
    w = _workload([40000], [[5, 6, 7], [9]], seed=stop, Hq=1, Hkv=1, W=32)
    g = Gpu(w, oracle_policy(16, fast=True, W=32), 16, 1)
    try:
        outcome = torch.full((1,), -9, dtype=torch.int32, device="cuda")
        began = time.perf_counter()
        ta.ta_ctx_selftest_exchange(g.ctx, 20_000_000, stop, outcome, g.stream)  # 20 ms
        torch.cuda.synchronize()
        assert time.perf_counter() - began < 1.0  # the limit that was given, not two seconds
        assert outcome.tolist() == [100 if stop == 4 else -9]
        assert g.poll() == (ta.TA_OK if stop == 4 else ta.TA_ERR_TIMEOUT)
        assert g.poll() == ta.TA_OK
    finally:
        g.close()
    _check(w, 16, True)  # and the next search is right
