"""Forms of a decode step's input: many and long patterns, ids outside the vocabulary, a captured step."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_11288_b200 as ta
from test_gpu_stream import _run
from test_gpu_stream_parts import SHARED, VOCAB, _state

pytestmark = pytest.mark.gpu


def test_many_and_long_patterns():
    # 70 patterns (three rounds of a lane per pattern) of 1 to 8 ids; suffixes of one another (the longest wins) and copies (the
    # lowest index wins); a budget of its own names the pattern that won
    rng = np.random.default_rng(9)
    ids = []
    for p in range(70):
        if p % 7 == 6:
            ids.append(list(ids[p - 5]))  # a copy: the earlier one wins
        elif p % 7 == 5:
            ids.append(ids[p - 1][-(1 + p % 4):])
        else:
            ids.append([int(x) for x in rng.integers(12, 60, 1 + (p * 5) % 8)])
    pats = oracle.Patterns(ids, budget=[float(1 + p) for p in range(70)], span=[1 + (p * 11) % 64 for p in range(70)])
    pol = oracle.preset("SEC33", 48, vocab_size=64)
    ora = _run(K=48, L=2, B=3, Hkv=1, steps=420, pats=pats, pol=pol, seed=4, check_every=13)
    won = {int(b) - 1 for o in ora for b, _ in o.anchors.values()}
    assert any(p >= 64 for p in won) and any(32 <= p < 64 for p in won) and any(p < 32 for p in won)
    assert {len(ids[p]) for p in won} == set(range(1, 9))
    assert all(ids.index(ids[p]) == p for p in won)


def _steps(st, t, pol, ids, attn, patterns, expect):
    """Steps through ids [steps][B] with the same attention masses for all of a sequence's units. Returns what was evicted."""
    L, B, Hkv, K = st.n_layers, st.batch, st.Hkv, st.K
    ctx = ta.ta_ctx_create(0, ta.ta_stream_scratch_bytes(st))
    pats = ta.ta_patterns_create(ctx, patterns)
    ev = torch.empty((len(ids), L, B, Hkv), dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    try:
        for i in range(len(ids)):
            a = attn[i].view(1, B, 1, K + 1).expand(L, B, Hkv, K + 1).contiguous()
            ta.ta_stream_step(ctx, pats, pol, st, ids[i].contiguous(), a, ev[i], stream)
        assert ta.ta_ctx_poll(ctx) == expect
        return ev.cpu()
    finally:
        ta.ta_patterns_destroy(pats)
        ta.ta_ctx_destroy(ctx)


@pytest.mark.parametrize("lam", [0.0, 1.0])
def test_ids_outside_the_vocabulary(lam):
    L, B, Hkv, K, steps = 2, 3, 2, 12, 60
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    ids = torch.randint(0, 6, (steps, B), generator=g, device="cuda", dtype=torch.int32)
    attn = torch.rand((steps, B, K + 1), generator=g, device="cuda")
    outside = torch.zeros((steps, B), dtype=torch.bool, device="cuda")
    outside[5::20, 0] = outside[7::25, 1] = True  # (the third sequence has none; no more than a unit has room for)
    ids_out = torch.where(outside, torch.where(ids > 2, torch.full_like(ids, VOCAB), torch.full_like(ids, -7)), ids)
    pol = ta.ta_policy_default(ta.TA_PRESET_SEC33, K)
    pol.vocab_size, pol.lambda_ = VOCAB, lam
    if lam:
        pol.alpha = pol.beta = pol.gamma = pol.delta = 0.0  # all that counts is how often an id came: one outside never did
    st, t = _state(L, B, Hkv, K)
    ev = _steps(st, t, pol, ids_out, attn, [] if lam else [[3], [4, 5]], ta.TA_ERR_DEVICE_BOUNDS)
    for b in range(B):  # a sequence's units had the same inputs: what the first one told the others left them all alike
        per = {n: x.view(L, B, Hkv, *x.shape[1:])[:, b].reshape(L * Hkv, -1) for n, x in t.items() if n not in SHARED}
        assert all(torch.equal(x, x[:1].expand_as(x)) for x in per.values())
        assert torch.equal(ev[:, :, b].reshape(steps, -1), ev[:, :1, b, :1].reshape(steps, 1).expand(steps, L * Hkv))
        want = torch.bincount(ids[:, b][~outside[:, b]].long(), minlength=VOCAB).to(torch.int32)
        assert torch.equal(t["hist"][b], want)
    gone = ev[:, 0, :, 0]
    if lam:
        assert not any(bool(outside[p, b]) for b in range(B) for p in gone[:, b].tolist() if p >= 0)
    else:  # how often an id came does not count: the same as with ids of their own that no pattern has
        st2, t2 = _state(L, B, Hkv, K)
        own = torch.where(outside, 10 + torch.arange(steps, device="cuda", dtype=torch.int32)[:, None] % 30, ids)
        ev2 = _steps(st2, t2, pol, own, attn, [[3], [4, 5]], ta.TA_OK)
        assert torch.equal(ev, ev2)
        for n in ("pos", "slot", "A", "P", "V", "S", "next_slot", "n_seen", "anc_B", "anc_L"):
            assert torch.equal(t[n], t2[n]), n


@pytest.mark.parametrize("L,B,Hkv", [(1, 1, 1), (2, 5, 4), (40, 64, 8)])  # the last one: two launches a step
def test_a_captured_step_is_replayed(L, B, Hkv):
    K, before, replays = 6, 9, 12
    pol = ta.ta_policy_default(ta.TA_PRESET_SEC33, K)
    pol.vocab_size = VOCAB
    (st, t), (ref, tr) = _state(L, B, Hkv, K), _state(L, B, Hkv, K)
    ctx = ta.ta_ctx_create(0, ta.ta_stream_scratch_bytes(st))
    pats = ta.ta_patterns_create(ctx, [[3], [4, 5]])
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    draw = lambda: (torch.randint(0, 8, (B,), generator=g, device="cuda", dtype=torch.int32),  # noqa: E731
                    torch.rand((L * B * Hkv, K + 1), generator=g, device="cuda"))
    ev, ev_ref = (torch.full((L * B * Hkv,), -9, dtype=torch.int32, device="cuda") for _ in range(2))
    stream = torch.cuda.current_stream().cuda_stream
    try:
        for _ in range(before):  # until the units are full: cache_len no longer changes
            ids, attn = draw()
            ta.ta_stream_step(ctx, pats, pol, st, ids, attn, ev, stream)
            ta.ta_stream_step(ctx, pats, pol, ref, ids, attn, ev_ref, stream)
        ids_in, attn_in = draw()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            ta.ta_stream_step(ctx, pats, pol, st, ids_in, attn_in, ev, torch.cuda.current_stream().cuda_stream)
        for _ in range(replays):
            ids, attn = draw()
            ids_in.copy_(ids), attn_in.copy_(attn)
            graph.replay()
            ta.ta_stream_step(ctx, pats, pol, ref, ids, attn, ev_ref, stream)
            assert torch.equal(ev, ev_ref)
        assert ta.ta_ctx_poll(ctx) == ta.TA_OK
        for n in t:
            assert torch.equal(t[n], tr[n]), n
    finally:
        ta.ta_patterns_destroy(pats)
        ta.ta_ctx_destroy(ctx)
