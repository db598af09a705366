"""What the first unit of a sequence tells the sequence's other units in a decode step."""
import pytest
import torch

import paper_2604_11288_b200 as ta
from test_gpu_stream_parts import _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,B,Hkv,K", [(1, 1, 2, 4), (2, 2, 4, 300), (32, 16, 8, 64)])
def test_no_wait_runs_out_while_every_word_comes(L, B, Hkv, K):
    # every word is read and cleared by one thread, so that no other can miss it and wait until the limit
    st, t = _state(L, B, Hkv, K)
    pol = ta.ta_policy_default(ta.TA_PRESET_THEOREM, K)
    pol.vocab_size = t["hist"].shape[1]
    ctx = ta.ta_ctx_create(0, ta.ta_stream_scratch_bytes(st))
    pats = ta.ta_patterns_create(ctx, [[3], [4, 5]])
    ta.ta_ctx_set_wait_limit(ctx, 200_000_000)
    g = torch.Generator(device="cuda")
    g.manual_seed(K)
    stream = torch.cuda.current_stream().cuda_stream
    U, steps = L * B * Hkv, 400
    ids = torch.randint(0, 8, (steps, B), generator=g, device="cuda", dtype=torch.int32)
    attn = torch.rand((U, K + 1), generator=g, device="cuda")
    ev = torch.empty(U, dtype=torch.int32, device="cuda")
    try:
        for i in range(steps):
            ta.ta_stream_step(ctx, pats, pol, st, ids[i], attn, ev, stream)
        assert ta.ta_ctx_poll(ctx) == ta.TA_OK
        assert torch.equal(t["n_seen"], torch.full_like(t["n_seen"], steps))
        last = t["pos"].gather(1, torch.full((U, 1), st.cache_len - 1, dtype=torch.int64, device="cuda"))
        assert torch.equal(last, torch.full_like(last, steps - 1))  # the newest token is never the one that goes
    finally:
        ta.ta_patterns_destroy(pats)
        ta.ta_ctx_destroy(ctx)
