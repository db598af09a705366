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


class _Streams:
    """A context and a decode state of 2 layers, 3 sequences and 4 heads, which has run until its units were full."""

    L, B, Hkv, K = 2, 3, 4, 40

    def __init__(self, seed):
        self.st, self.t = _state(self.L, self.B, self.Hkv, self.K)
        self.U = self.L * self.B * self.Hkv
        self.vocab = self.t["hist"].shape[1]
        self.pol = ta.ta_policy_default(ta.TA_PRESET_SEC33, self.K)
        self.pol.vocab_size = self.vocab
        self.ctx = ta.ta_ctx_create(0, ta.ta_stream_scratch_bytes(self.st))
        self.pats = ta.ta_patterns_create(self.ctx, [[3], [4, 5]])
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        self.ev = torch.full((self.U,), -9, dtype=torch.int32, device="cuda")
        self.stream = torch.cuda.current_stream().cuda_stream
        self.first = torch.zeros(self.U, dtype=torch.bool)  # the first unit of every sequence
        self.first[: self.B * self.Hkv : self.Hkv] = True
        for _ in range(self.K + 7):
            self.step(*self.inputs())

    def inputs(self):
        ids = torch.randint(0, 8, (self.B,), generator=self.g, device="cuda", dtype=torch.int32)
        return ids, torch.rand((self.U, self.K + 1), generator=self.g, device="cuda")

    def step(self, ids, attn):
        ta.ta_stream_step(self.ctx, self.pats, self.pol, self.st, ids, attn, self.ev, self.stream)

    def timed_out_step(self, ids, attn):
        ta.ta_ctx_selftest_step_wait(self.ctx, self.pats, self.pol, self.st, ids, attn, self.ev, 1_000_000, self.stream)

    def state(self):
        torch.cuda.synchronize()
        return {**{n: x.cpu().clone() for n, x in self.t.items()}, "ev": self.ev.cpu().clone()}

    def restore(self, s):
        for n, x in self.t.items():
            x.copy_(s[n])
        self.ev.copy_(s["ev"])
        torch.cuda.synchronize()

    def close(self):
        ta.ta_patterns_destroy(self.pats)
        ta.ta_ctx_destroy(self.ctx)


def _same(a, b, units=None):
    for n in a:
        x, y = a[n], b[n]
        if units is not None:
            if n in ("n_seen", "hist", "tok_ring", "anc_B", "anc_L"):
                continue  # of a sequence, not of a unit
            x, y = x[units], y[units]
        if not torch.equal(x, y):
            return False
    return True


@pytest.fixture
def streams():
    s, ref = _Streams(5), _Streams(5)
    try:
        yield s, ref
    finally:
        s.close()
        ref.close()


def test_a_unit_whose_wait_runs_out_keeps_its_state(streams):
    s, ref = streams
    before = s.state()
    ids, attn = s.inputs()
    s.timed_out_step(ids, attn)
    after = s.state()
    assert _same(before, after, ~s.first)
    ref.step(*ref.inputs())
    assert _same(ref.state(), after, s.first)  # the first units had all that they need
    # until the context is polled nothing more happens to any unit
    s.step(*s.inputs())
    assert _same(after, s.state())
    assert ta.ta_ctx_poll(s.ctx) == ta.TA_ERR_TIMEOUT
    assert ta.ta_ctx_poll(s.ctx) == ta.TA_OK


def test_words_that_came_late_are_not_taken_for_the_next_steps(streams):
    s, ref = streams
    before = s.state()
    s.timed_out_step(*s.inputs())
    assert ta.ta_ctx_poll(s.ctx) == ta.TA_ERR_TIMEOUT
    s.restore(before)
    s.g.manual_seed(77), ref.g.manual_seed(77)
    for _ in range(5):
        s.step(*s.inputs()), ref.step(*ref.inputs())
        assert _same(ref.state(), s.state())
    assert ta.ta_ctx_poll(s.ctx) == ta.TA_OK


def test_late_words_are_cleared_whatever_was_reported_first(streams):
    s, ref = streams
    before = s.state()
    ids, attn = s.inputs()
    s.step(torch.full_like(ids, s.vocab), attn)  # outside the vocabulary: the first thing that is reported
    s.timed_out_step(ids, attn)
    assert ta.ta_ctx_poll(s.ctx) == ta.TA_ERR_TIMEOUT  # what has cost the state comes before what has not
    s.restore(before)
    s.g.manual_seed(78), ref.g.manual_seed(78)
    for _ in range(5):
        s.step(*s.inputs()), ref.step(*ref.inputs())
        assert _same(ref.state(), s.state())
    assert ta.ta_ctx_poll(s.ctx) == ta.TA_OK


def test_a_poll_returns_when_its_clearing_is_complete(streams):
    # the step after it is on a stream that does not wait for the legacy stream's work
    s, ref = streams
    own = torch.cuda.Stream()
    s.stream = own.cuda_stream
    for i in range(30):
        before = s.state()
        s.timed_out_step(*s.inputs())
        torch.cuda.synchronize()
        s.restore(before)
        s.g.manual_seed(100 + i), ref.g.manual_seed(100 + i)
        inputs = s.inputs()
        polled, idle = ta.ta_ctx_poll(s.ctx), torch.cuda.default_stream().query()
        s.step(*inputs)
        assert polled == ta.TA_ERR_TIMEOUT and idle
        ref.step(*ref.inputs())
        assert _same(ref.state(), s.state())
    assert ta.ta_ctx_poll(s.ctx) == ta.TA_OK


def test_a_time_out_of_another_call_does_not_concern_the_step(streams):
    s, ref = streams
    ta.ta_ctx_selftest_wait(s.ctx, 1_000_000, torch.zeros(1, dtype=torch.int32, device="cuda"), s.stream)
    for _ in range(5):
        s.step(*s.inputs()), ref.step(*ref.inputs())
    assert _same(ref.state(), s.state())
    assert ta.ta_ctx_poll(s.ctx) == ta.TA_ERR_TIMEOUT
    assert ta.ta_ctx_poll(ref.ctx) == ta.TA_OK


@pytest.mark.parametrize("limit", [0, 1_000_000_001])
def test_the_self_tests_limit_is_checked(streams, limit):
    s, _ = streams
    with pytest.raises(ta.TAError) as e:
        ta.ta_ctx_selftest_step_wait(s.ctx, s.pats, s.pol, s.st, s.ev, s.ev, s.ev, limit, s.stream)
    assert e.value.status == ta.TA_ERR_INVALID_ARG


def test_the_self_test_holds_no_longer_than_the_units_wait():
    # a call of several launches, and one in which nobody waits: held once, or not at all
    for L, B, Hkv, expect in ((2, 9000, 2, ta.TA_ERR_TIMEOUT), (1, 20000, 1, ta.TA_OK)):
        st, t = _state(L, B, Hkv, 4)
        pol = ta.ta_policy_default(ta.TA_PRESET_THEOREM, 4)
        pol.vocab_size = t["hist"].shape[1]
        ctx = ta.ta_ctx_create(0, ta.ta_stream_scratch_bytes(st))
        pats = ta.ta_patterns_create(ctx, [[3]])
        stream = torch.cuda.current_stream().cuda_stream
        ids = torch.randint(0, 8, (B,), device="cuda", dtype=torch.int32)
        try:
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            ta.ta_ctx_selftest_step_wait(ctx, pats, pol, st, ids, torch.rand((L * B * Hkv, 5), device="cuda"),
                                         torch.empty(L * B * Hkv, dtype=torch.int32, device="cuda"), 50_000_000, stream)
            e1.record()
            assert ta.ta_ctx_poll(ctx) == expect
            assert e0.elapsed_time(e1) < (300 if expect else 50)
        finally:
            ta.ta_patterns_destroy(pats)
            ta.ta_ctx_destroy(ctx)
