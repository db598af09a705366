"""The calls whose speed matters to a program that uses this library, as measurable cases.

A case is a plain dict. `path` names the entry point and `mode` the scoring; the other fields are its sizes:

  compress   ta_compress, all layers of a batch in one call (after prefill)
  layers     ta_compress once per layer under one epoch (a prefill that compacts each layer as soon as it is done)
  lse        ta_compress_lse, the prefill kernel's log-sum-exp of the window rows at hand
  scores     ta_compress_scores, another method's importance scores in place of the attention terms
  host       ta_compress_host, the cache offloaded to pinned host memory
  decode     ta_stream_step, one eviction decision per unit and generated token, caches full
  detect     ta_detect_embedding and ta_sponsor_mask_conf, anchors found by embedding similarity

Sizes follow the configurations of ta_workloads (paper-style 4096-token prompts up to 16 x 32768 and 4 x 131072 tokens)
with fewer layers per call where three copies of the inputs would not fit the card. Token ids are uniform over the
vocabulary with anchor patterns planted at random depths; queries, keys and values are N(0, 1) in bf16.
"""
import math
import random

import numpy as np
import torch

import paper_2604_11288_b200 as ta

D = 128        # head_dim
VOCAB = 32000
DEV = "cuda:0"
PATTERN_LENS = (1, 1, 2, 2, 2, 3, 3, 3)
CONCEPTS = 8

# ------------------------------------------------------------------------------------------------ the cases


def listed():
    return [
        # one layer of one 4096-token prompt: the smallest call, paid per layer by a program that does not batch layers
        dict(name="layer_4k", path="compress", mode="scored", layers=1, batch=1, n_lo=4096, n_hi=4096, heads=32, kv=8,
             window=32, keep=16, spans=4),
        # one 4096-token prompt, every layer of the model at once, the paper's headline budget
        dict(name="prompt_4k", path="compress", mode="scored", layers=32, batch=1, n_lo=4096, n_hi=4096, heads=32, kv=8,
             window=32, keep=16, spans=1),
        # the same prompt without attention scores (TA-Fast) at the largest budget of the sweep
        dict(name="prompt_4k_fast", path="compress", mode="fast", layers=32, batch=1, n_lo=4096, n_hi=4096, heads=32,
             kv=8, window=32, keep=1024, spans=1),
        # throughput serving: 16 long prompts, a 64-query window, half of a 32-layer model per call
        dict(name="batch_32k", path="compress", mode="scored", layers=16, batch=16, n_lo=32768, n_hi=32768, heads=32,
             kv=8, window=64, keep=2048, spans=64),
        # very long contexts without attention scores: mask, selection and gather only
        dict(name="batch_131k_fast", path="compress", mode="fast", layers=16, batch=4, n_lo=131072, n_hi=131072,
             heads=32, kv=8, window=32, keep=4096, spans=512),
        # an agent server's ragged batch: 64 conversations of very different lengths, a small budget each
        dict(name="ragged_agents", path="compress", mode="scored", layers=8, batch=64, n_lo=2048, n_hi=16384, heads=32,
             kv=8, window=32, keep=64, spans=8),
        # layer by layer during prefill on one shard of a tensor-parallel model, prompts of odd lengths
        dict(name="shard_by_layer", path="layers", mode="scored", layers=32, batch=4, n_lo=1500, n_hi=7000, heads=8, kv=2,
             window=32, keep=128, spans=4),
        # the prefill attention kernel has left the normalisers: one pass over the keys, a length that fills no tile
        dict(name="prompt_8k_lse", path="lse", mode="scored", layers=32, batch=1, n_lo=8111, n_hi=8111, heads=32, kv=8,
             window=32, keep=256, spans=4),
        # sponsorship on top of another eviction score, ragged batch
        dict(name="ragged_scores", path="scores", mode="scored", layers=32, batch=8, n_lo=1000, n_hi=8000, heads=32, kv=8,
             window=32, keep=512, spans=8),
        # a cache that was offloaded to host memory
        dict(name="offloaded_3k", path="host", mode="scored", layers=8, batch=2, n_lo=3000, n_hi=3000, heads=32, kv=8,
             window=32, keep=128, spans=4),
        # the decode loop of 16 sequences with 256 cached tokens per head
        dict(name="decode_256", path="decode", mode="scored", layers=32, batch=16, n_lo=4096, n_hi=4096, heads=32, kv=8,
             window=32, keep=256, spans=16),
        # anchors by embedding similarity over a batch of long prompts, 2048-wide input embeddings
        dict(name="detect_2048", path="detect", mode="fast", layers=1, batch=4, n_lo=32768, n_hi=32768, heads=2048, kv=8,
             window=32, keep=64, spans=64),
    ]


# what each path of draw() may reach; nothing drawn moves or computes more than the largest listed case does
MAX_CACHE_BYTES = 16 * 16 * 32768 * 8 * D * 2 * 2
MAX_SCORES = 16 * 16 * 32768 * 8 * 256
RANGES = {  # path: (tokens per sequence, sequences, layers, kept tokens, share of the draws)
    "compress": ((1024, 131072), (1, 64), (1, 32), (16, 4096), 6),
    "layers": ((1024, 16384), (1, 8), (8, 32), (16, 1024), 1),
    "lse": ((1024, 16384), (1, 4), (4, 32), (16, 1024), 1),
    "scores": ((1024, 16384), (1, 16), (4, 32), (16, 2048), 1),
    "host": ((1024, 8192), (1, 4), (1, 8), (16, 512), 1),
    "decode": ((4096, 4096), (1, 32), (8, 32), (64, 2048), 1),
    "detect": ((2048, 32768), (1, 8), (1, 1), (64, 64), 1),
}


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    paths = list(RANGES)
    path = rng.choices(paths, [RANGES[p][4] for p in paths])[0]
    tokens, seqs, depth, keep, _ = RANGES[path]
    mode = "fast" if path == "detect" or (path == "compress" and rng.random() < 0.35) else "scored"
    heads, kv = rng.choice([(32, 8), (32, 8), (8, 2), (16, 4), (8, 8), (16, 2)])
    if path == "detect":
        heads = 32 * rng.randint(32, 128)  # the embedding width
    window = rng.choice([16, 32, 32, 64]) if path != "detect" and heads // kv <= 4 else 32
    n, batch, layers = _log_int(rng, *tokens), _log_int(rng, *seqs), _log_int(rng, *depth)
    ragged = batch > 1 and path not in ("lse", "host", "decode", "detect") and rng.random() < 0.5
    per = layers * n * kv
    while batch > 1 and (batch * per * D * 4 > MAX_CACHE_BYTES or batch * per * (heads // kv) * window > MAX_SCORES):
        batch -= 1
    return dict(path=path, mode=mode, layers=layers, batch=batch, n_lo=max(512, n // 4) if ragged and batch > 1 else n,
                n_hi=n, heads=heads, kv=kv, window=window, keep=min(_log_int(rng, *keep), n // 2),
                spans=rng.choice([1, 4, 16, 64]))


# ------------------------------------------------------------------------------------------------ inputs


def _lengths(case):
    """Tokens of every sequence; a ragged batch's lengths are the same whatever the seed of the inputs."""
    lo, hi, b = case["n_lo"], case["n_hi"], case["batch"]
    rng = random.Random(1000003 * lo + 1009 * hi + b)
    return [hi if lo == hi else rng.randint(lo, hi) for _ in range(b)]


def _token_ids(case, lengths, rng):
    """Uniform ids with planted anchors: every sequence is cut into `spans` slots, one pattern at a random place in each."""
    pats, at = [], 0
    ids_of = rng.choice(VOCAB, size=sum(PATTERN_LENS), replace=False)
    for ln in PATTERN_LENS:
        pats.append([int(t) for t in ids_of[at:at + ln]])
        at += ln
    ids = rng.integers(0, VOCAB, size=sum(lengths)).astype(np.int32)
    base = 0
    for n in lengths:
        slot = n // case["spans"]
        if slot > 32:
            for s in range(case["spans"]):
                p = pats[int(rng.integers(0, len(pats)))]
                i = base + s * slot + int(rng.integers(0, slot - 30))
                ids[i:i + len(p)] = p
        base += n
    return ids, pats


class State:
    """A caller's long-lived objects (context, patterns, policy) and one set of inputs and output buffers."""
    ctx = pats = None

    def __del__(self):
        if self.pats is not None:
            ta.ta_patterns_destroy(self.pats)
        if self.ctx is not None:
            ta.ta_ctx_destroy(self.ctx)


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    s = State()
    s.case, s.path, s.fast = case, case["path"], case["mode"] == "fast"
    s.L, s.B, s.Hq, s.Hkv, s.K = case["layers"], case["batch"], case["heads"], case["kv"], case["keep"]
    lengths = _lengths(case)
    s.total, s.uniform = sum(lengths), case["n_lo"] == case["n_hi"]
    ids, pats = _token_ids(case, lengths, rng)
    s.policy = ta.ta_policy_default(ta.TA_PRESET_THEOREM, s.K)
    s.policy.obs_window = case["window"]
    s.policy.mode = ta.TA_MODE_FAST if s.fast else ta.TA_MODE_SCORED
    s.policy.vocab_size = VOCAB
    if s.path == "decode":
        _prepare_decode(s, ids, pats, g, rng)
        return s
    s.ids = torch.from_numpy(ids).to(DEV)
    s.cu = None
    if not s.uniform:
        s.cu = torch.tensor(np.concatenate([[0], np.cumsum(lengths)]), dtype=torch.int32, device=DEV)
    s.batch = ta.make_batch(1 if s.path == "layers" else s.L, s.B, lengths[0] if s.uniform else 0, max(lengths), s.total,
                            s.cu)
    s.ctx = ta.ta_ctx_create(0, ta.ta_scratch_bytes(s.batch, s.Hq, s.Hkv, D, s.K, s.policy))
    s.pats = ta.ta_patterns_create(s.ctx, pats)
    if s.path == "detect":
        _prepare_detect(s, g)
        return s
    kv_shape = (s.L, s.B, s.Hkv, lengths[0], D) if s.uniform else (s.L, s.Hkv, s.total, D)
    bf16 = dict(dtype=torch.bfloat16, device=DEV)
    s.k = torch.randn(kv_shape, generator=g, **bf16)
    s.v = torch.randn(kv_shape, generator=g, **bf16)
    s.q = None
    if not s.fast and s.path != "scores":
        s.q = torch.randn((s.L, s.B, s.Hq, case["window"], D), generator=g, **bf16)
    s.k_out = torch.empty((s.L, s.B, s.Hkv, s.K, D), **bf16)
    s.v_out = torch.empty((s.L, s.B, s.Hkv, s.K, D), **bf16)
    s.idx = torch.empty((s.L, s.B, s.Hkv, s.K), dtype=torch.int32, device=DEV)
    s.count = torch.empty((s.L, s.B, s.Hkv), dtype=torch.int32, device=DEV)
    if s.path == "lse":
        s.lse = _window_lse(s, lengths[0], case["window"])
    elif s.path == "scores":
        # accumulated attention per token: positive, heavy-tailed, mean one
        s.score = torch.empty((s.L, s.Hkv, s.total), dtype=torch.float32, device=DEV).exponential_(generator=g)
    elif s.path == "layers":
        s.epoch = 0
    elif s.path == "host":
        _prepare_host(s)
    # the retained rows are copies: they are compared as bits
    s.out = {"idx": s.idx, "count": s.count, "k_rows": s.k_out.view(torch.int16), "v_rows": s.v_out.view(torch.int16)}
    return s


def _window_lse(s, n, w):
    """Natural-log softmax normalisers [L][B][Hq][W] of the window rows, as a prefill attention kernel leaves them."""
    lse = torch.empty((s.L, s.B, s.Hq, w), dtype=torch.float32, device=DEV)
    hidden = torch.arange(n, device=DEV).view(1, -1) > torch.arange(n - w, n, device=DEV).view(-1, 1)
    for layer in range(s.L):
        for b in range(s.B):
            k = s.k[layer, b].float().repeat_interleave(s.Hq // s.Hkv, dim=0)
            x = torch.bmm(s.q[layer, b].float(), k.transpose(1, 2)) / math.sqrt(D)
            lse[layer, b] = torch.logsumexp(x.masked_fill(hidden, float("-inf")), dim=-1)
    return lse


def _prepare_host(s):
    """Moves inputs and outputs to pinned host memory and lends a device workspace."""
    pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)  # noqa: E731
    s.ids, s.q, s.k, s.v = pin(s.ids), pin(s.q), pin(s.k), pin(s.v)
    s.k_out, s.v_out, s.idx, s.count = pin(s.k_out), pin(s.v_out), pin(s.idx), pin(s.count)
    s.ws_bytes = ta.ta_compress_host_workspace_bytes(s.batch, s.Hq, s.Hkv, D, s.K, s.policy)
    s.ws = torch.empty(s.ws_bytes, dtype=torch.uint8, device=DEV)


def _prepare_detect(s, g):
    """Input embeddings (`heads` wide), the concepts, and every planted anchor's embedding near one of the concepts."""
    width = s.Hq
    s.emb = torch.randn((s.total, width), generator=g, dtype=torch.bfloat16, device=DEV)
    s.concepts = torch.randn((CONCEPTS, width), generator=g, dtype=torch.bfloat16, device=DEV)
    n_near = s.B * s.case["spans"]
    near = torch.randperm(s.total, generator=g, device=DEV)[:n_near]
    which = torch.randint(0, CONCEPTS, (near.numel(),), generator=g, device=DEV)
    s.emb[near] = s.concepts[which] + 0.5 * s.emb[near]
    s.conf = torch.empty(s.total, dtype=torch.float32, device=DEV)
    s.flags = torch.empty(s.total, dtype=torch.uint8, device=DEV)
    s.voucher = torch.empty(s.total, dtype=torch.float32, device=DEV)
    s.u_static = torch.empty(s.total, dtype=torch.float32, device=DEV)
    s.out = {"conf": s.conf, "flags": s.flags, "voucher": s.voucher, "u_static": s.u_static}


DECODE_INPUTS = 8  # steps' tokens and attention masses held ready, taken in turn


def _prepare_decode(s, ids, pats, g, rng):
    """Full caches behind a prompt: K retained positions per unit, in order, with their rows in arbitrary cache slots."""
    n, U, C = s.case["n_hi"], s.L * s.B * s.Hkv, s.K + 1
    dev_ids = torch.from_numpy(ids).to(DEV).view(s.B, n)
    rows = torch.rand((U, n), generator=g, device=DEV).topk(s.K, dim=1).indices.sort(dim=1).values.to(torch.int32)
    seq = (torch.arange(U, device=DEV) // s.Hkv) % s.B
    t = {}
    t["pos"] = torch.zeros((U, C), dtype=torch.int32, device=DEV)
    t["pos"][:, :s.K] = rows
    t["slot"] = torch.rand((U, C), generator=g, device=DEV).argsort(dim=1).to(torch.int32)
    t["next_slot"] = t["slot"][:, s.K].contiguous()  # the one row that holds no token
    t["tok"] = torch.zeros((U, C), dtype=torch.int32, device=DEV)
    t["tok"][:, :s.K] = dev_ids[seq].gather(1, rows.long())
    t["A"] = torch.empty((U, C), dtype=torch.float32, device=DEV).exponential_(generator=g)
    t["P"] = 0.1 * torch.rand((U, C), generator=g, device=DEV)
    sponsored = torch.rand((U, C), generator=g, device=DEV) < 0.05
    t["V"] = torch.where(sponsored, 15.0 * torch.rand((U, C), generator=g, device=DEV), torch.zeros((), device=DEV))
    t["S"] = (torch.rand((U, C), generator=g, device=DEV) < 0.02).to(torch.uint8)
    t["n_seen"] = torch.full((s.B,), n, dtype=torch.int32, device=DEV)
    t["hist"] = torch.zeros((s.B, VOCAB), dtype=torch.int32, device=DEV)
    t["hist"].scatter_add_(1, dev_ids.long(), torch.ones_like(dev_ids))
    last = torch.arange(n - 8, n, device=DEV)
    t["tok_ring"] = torch.zeros((s.B, 8), dtype=torch.int32, device=DEV)
    t["tok_ring"][:, last % 8] = dev_ids[:, last]
    t["anc_B"] = torch.zeros((s.B, 64), dtype=torch.float32, device=DEV)
    t["anc_L"] = torch.zeros((s.B, 64), dtype=torch.int32, device=DEV)
    s.tensors = t
    s.stream_state = ta.ta_stream()
    st = s.stream_state
    st.n_layers, st.batch, st.Hkv, st.K, st.cache_len = s.L, s.B, s.Hkv, s.K, s.K
    for name, x in t.items():
        setattr(st, name, x.data_ptr())
    s.ctx = ta.ta_ctx_create(0, ta.ta_stream_scratch_bytes(st))
    s.pats = ta.ta_patterns_create(s.ctx, pats)
    new = rng.integers(0, VOCAB, size=(DECODE_INPUTS, s.B)).astype(np.int32)
    new[3] = pats[0][0]  # now and then a generated token is an anchor
    s.new_ids = torch.from_numpy(new).to(DEV)
    s.attn = torch.rand((DECODE_INPUTS, U, C), generator=g, device=DEV)
    s.attn /= s.attn.sum(dim=2, keepdim=True)
    s.evicted = torch.empty(U, dtype=torch.int32, device=DEV)
    s.step = 0
    s.out = {"evicted": s.evicted, **{k: t[k] for k in ("pos", "slot", "tok", "A", "P", "V", "S", "next_slot", "n_seen")}}


# ------------------------------------------------------------------------------------------------ one pass


def run(s):
    stream = torch.cuda.current_stream().cuda_stream
    ragged = not s.uniform
    if s.path == "compress":
        ta.ta_compress(s.ctx, s.pats, s.policy, s.batch, s.Hq, s.Hkv, D, s.K, s.ids, ta.view(s.q), ta.view(s.k, ragged),
                       ta.view(s.v, ragged), 0, s.k_out, s.v_out, s.idx, s.count, stream)
    elif s.path == "layers":
        s.epoch += 1  # a new batch of prompts; its layers share the per-sequence work
        for i in range(s.L):
            one = slice(i, i + 1)
            ta.ta_compress(s.ctx, s.pats, s.policy, s.batch, s.Hq, s.Hkv, D, s.K, s.ids, ta.view(s.q[one]),
                           ta.view(s.k[one], ragged), ta.view(s.v[one], ragged), s.epoch, s.k_out[i], s.v_out[i],
                           s.idx[i], s.count[i], stream)
    elif s.path == "lse":
        ta.ta_compress_lse(s.ctx, s.pats, s.policy, s.batch, s.Hq, s.Hkv, D, s.K, s.ids, ta.view(s.q), ta.view(s.k),
                           ta.view(s.v), s.lse, 0, s.k_out, s.v_out, s.idx, s.count, stream)
    elif s.path == "scores":
        ta.ta_compress_scores(s.ctx, s.pats, s.policy, s.batch, s.Hkv, D, s.K, s.ids, s.score, None,
                              ta.view(s.k, ragged), ta.view(s.v, ragged), 0, s.k_out, s.v_out, s.idx, s.count, stream)
    elif s.path == "host":
        ta.ta_compress_host(s.ctx, s.pats, s.policy, s.batch, s.Hq, s.Hkv, D, s.K, s.ids, s.q, s.k, s.v, s.k_out, s.v_out,
                            s.idx, s.count, s.ws, s.ws_bytes, stream)
    elif s.path == "decode":
        i = s.step % DECODE_INPUTS
        s.step += 1
        ta.ta_stream_step(s.ctx, s.pats, s.policy, s.stream_state, s.new_ids[i], s.attn[i], s.evicted, stream)
    else:
        ta.ta_detect_embedding(s.ctx, s.total, s.emb, s.Hq, s.Hq, s.concepts, CONCEPTS, s.conf, stream)
        ta.ta_sponsor_mask_conf(s.ctx, s.policy, s.batch, s.ids, s.conf, 0.3, 15.0, 6, 0, s.flags, s.voucher,
                                s.u_static, stream)
    return s.out


# ------------------------------------------------------------------------------------------------ what a pass costs


def work(case):
    L, B, Hq, Hkv, K, W = (case[k] for k in ("layers", "batch", "heads", "kv", "keep", "window"))
    lengths = _lengths(case)
    total = sum(lengths)
    path = case["path"]
    if path == "decode":
        # 25 bytes of state per cached token read and written, its attention mass read
        return {"bytes": L * B * Hkv * (K + 1) * (2 * 25 + 4), "flops": 0}
    if path == "detect":
        # embeddings and ids in; confidence, flag, voucher and utility out
        return {"bytes": total * (2 * Hq + 4 + 4 + 1 + 4 + 4), "flops": 2 * total * Hq * CONCEPTS}
    rows = L * Hkv * sum(min(K, n) for n in lengths)  # retained, of each of K and V
    out = L * B * Hkv * (K * (2 * 2 * D + 4) + 4)
    if case["mode"] == "fast":
        return {"bytes": total * 4 + rows * 2 * 2 * D + out, "flops": 0}
    if path == "scores":
        return {"bytes": total * 4 + L * Hkv * total * 4 + rows * 2 * 2 * D + out, "flops": 0}
    # every key once (the retained ones among them), the retained values
    return {"bytes": total * 4 + L * B * Hq * W * 2 * D + L * Hkv * total * 2 * D + rows * 2 * D + out,
            "flops": 2 * L * Hq * W * D * total}


def tolerance(case):
    if case["path"] == "detect":
        return {"rel": 2e-5}  # fp32 sums of a few thousand bf16 products; flags are exact
    if case["mode"] == "fast" or case["path"] in ("scores", "decode"):
        return "exact"  # fp32 with one rounding per operation decides the selection
    # attention terms are fp32 sums of exponentials: tokens whose utilities tie to the last bits may change places at
    # the edge of the budget, and every retained row behind such a place moves by one
    return {"rel": 0.0, "differ": 0.01}
