"""Decode steps between the calls of one epoch: the step has no part in the per-sequence results that the context keeps for them."""
import pytest
import torch

import paper_2604_11288_b200 as ta
import ta_workloads as tw
from ta_testlib import Gpu, oracle_policy
from test_gpu_stream_parts import _state

pytestmark = pytest.mark.gpu


def test_a_decode_step_leaves_the_epochs_results():
    w = tw.config1(n=1500, Hq=8, Hkv=2)
    K = 24
    Q, Kc, Vc = (x.cuda() for x in tw.make_qkv(w, [0]))
    g = Gpu(w, oracle_policy(K, "THEOREM", W=w.W), K, 1)
    st, t = _state(1, 3, 2, 8)
    pol = ta.ta_policy_default(ta.TA_PRESET_THEOREM, 8)
    pol.vocab_size = t["hist"].shape[1]
    try:
        def compress():
            out = g.compress(Q, Kc, Vc, epoch=7)
            return out, ta.ta_ctx_last_launch_info(g.ctx)[3]

        whole, n_whole = compress()
        again, n_again = compress()
        assert n_again < n_whole
        ta.ta_stream_step(g.ctx, g.pats, pol, st, torch.ones(3, dtype=torch.int32, device="cuda"),
                          torch.rand(6, 9, device="cuda"), torch.empty(6, dtype=torch.int32, device="cuda"), g.stream)
        after, n_after = compress()
        assert g.poll() == ta.TA_OK
        assert n_after == n_again
        for a, b, c in zip(whole, again, after):
            assert torch.equal(a, b) and torch.equal(a, c)
    finally:
        g.close()
