"""A decode step of more units than one launch has words for is enqueued in parts (of layers, of sequences or of heads): the same
state after several steps, bit for bit, as when pieces that one launch holds are stepped alone with a copy of what the sequences
share."""
import numpy as np
import pytest
import torch

import paper_2604_11288_b200 as ta

pytestmark = pytest.mark.gpu
VOCAB = 40


def _state(L, B, Hkv, K):
    U, C = L * B * Hkv, K + 1
    z = lambda shape, dt: torch.zeros(shape, dtype=dt, device="cuda")  # noqa: E731
    t = {n: z((U, C), torch.int32) for n in ("pos", "slot", "tok")}
    t.update({n: z((U, C), torch.float32) for n in ("A", "P", "V")})
    t.update(S=z((U, C), torch.uint8), next_slot=z(U, torch.int32), n_seen=z(B, torch.int32), hist=z((B, VOCAB), torch.int32),
             tok_ring=z((B, 8), torch.int32), anc_B=z((B, 64), torch.float32), anc_L=z((B, 64), torch.int32))
    st = ta.ta_stream()
    st.n_layers, st.batch, st.Hkv, st.K, st.cache_len = L, B, Hkv, K, 0
    for name, x in t.items():
        setattr(st, name, x.data_ptr())
    return st, t


SHARED = ("n_seen", "hist", "tok_ring", "anc_B", "anc_L")  # of a sequence, the others of a unit
WORDS = 16384  # units of one launch


def _pieces(L, B, Hkv):
    """(layer, first and last sequence, first and last head) of pieces that one launch each can hold."""
    ng = min(Hkv, WORDS)
    nb = min(B, WORDS // ng)
    return [(l, b, min(b + nb, B), g, min(g + ng, Hkv)) for l in range(L) for b in range(0, B, nb) for g in range(0, Hkv, ng)]


# cut by sequence (the last part smaller), by sequence within a layer, by layer (32 and 8), by head (16384 and 616)
@pytest.mark.parametrize("L,B,Hkv", [(3, 1500, 16), (2, 66000, 1), (40, 64, 8), (2, 3, 17000)])
def test_parts_leave_the_state_of_single_layers(L, B, Hkv):
    K, steps = 5, 14
    pol = ta.ta_policy_default(ta.TA_PRESET_THEOREM, K)
    pol.vocab_size = VOCAB
    assert L * B * Hkv > WORDS
    whole, tw = _state(L, B, Hkv, K)
    pieces = _pieces(L, B, Hkv)
    assert all((b1 - b0) * (g1 - g0) <= WORDS for _, b0, b1, g0, g1 in pieces)
    single = [_state(1, b1 - b0, g1 - g0, K) for _, b0, b1, g0, g1 in pieces]
    ctx = ta.ta_ctx_create(0, ta.ta_stream_scratch_bytes(whole))
    pats = ta.ta_patterns_create(ctx, [[3], [4, 5]])
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    stream = torch.cuda.current_stream().cuda_stream
    try:
        for _ in range(steps):
            ids = torch.randint(0, 8, (B,), generator=g, device="cuda", dtype=torch.int32)
            attn = torch.rand((L, B, Hkv, K + 1), generator=g, device="cuda")
            ev = torch.full((L, B, Hkv), -9, dtype=torch.int32, device="cuda")
            ta.ta_stream_step(ctx, pats, pol, whole, ids, attn, ev, stream)
            for (l, b0, b1, g0, g1), (st, _) in zip(pieces, single):
                e1 = torch.full((b1 - b0, g1 - g0), -9, dtype=torch.int32, device="cuda")
                ta.ta_stream_step(ctx, pats, pol, st, ids[b0:b1].contiguous(), attn[l, b0:b1, g0:g1].contiguous(), e1, stream)
                assert torch.equal(e1, ev[l, b0:b1, g0:g1])
        assert ta.ta_ctx_poll(ctx) == ta.TA_OK
        for (l, b0, b1, g0, g1), (_, t1) in zip(pieces, single):
            for name, x in t1.items():
                y = tw[name]
                y = y[b0:b1] if name in SHARED else y.view(L, B, Hkv, *y.shape[1:])[l, b0:b1, g0:g1].reshape(x.shape)
                np.testing.assert_array_equal(x.cpu().numpy(), y.cpu().numpy(), err_msg=f"layer {l} sequences {b0} heads {g0} {name}")
    finally:
        ta.ta_patterns_destroy(pats)
        ta.ta_ctx_destroy(ctx)
