"""The decode step at the largest budgets, nine cached tokens per thread: a few steps from a full state against the streaming oracle."""
import numpy as np
import pytest
import torch

import oracle
from oracle.ta_stream_oracle import StreamOracle
from test_gpu_stream import GpuStream

pytestmark = pytest.mark.gpu


# the smallest unit of nine tokens per thread, a whole number of warps, one token more, and the largest units
@pytest.mark.parametrize("K", [2048, 2303, 2304, 4095, 4096])
@pytest.mark.parametrize("sponsored", [0.01, 0.6])
def test_steps_of_a_full_state(K, sponsored):
    rng = np.random.default_rng(K)
    pats = oracle.Patterns([[3], [4, 5]], budget=[15.0, 2.0], span=[5, 9])
    pol = oracle.preset("SEC33", K, vocab_size=64)
    U, n = 2, K + 300  # tokens seen, of which K are cached
    g = GpuStream(pats, pol, K, 1, 1, U)
    ora = StreamOracle(pats, pol, K, U)
    try:
        ora.ids = [int(x) for x in rng.integers(0, 40, n)]
        host = {k: v.cpu().numpy() for k, v in g.t.items()}
        for u, un in enumerate(ora.units):
            pos = np.sort(rng.choice(n, K, replace=False))
            slot = rng.permutation(K + 1)
            A, P = rng.random((2, K)).astype(np.float32)
            V = np.where(rng.random(K) < sponsored, rng.integers(1, 200, K), 0).astype(np.float32) / np.float32(64)  # ties among them
            S = (rng.random(K) < 0.1).astype(np.uint8)
            un.pos, un.S = [int(p) for p in pos], [int(x) for x in S]
            un.A, un.P, un.V = [list(x) for x in (A, P, V)]
            for name, x in (("pos", pos), ("slot", slot[:K]), ("tok", [ora.ids[p] for p in pos]), ("A", A), ("P", P), ("V", V), ("S", S)):
                host[name][u, :K] = x
            host["next_slot"][u] = slot[K]
        host["n_seen"][0] = n
        host["hist"][0] = np.bincount(ora.ids, minlength=64)
        for p in range(n - 8, n):
            host["tok_ring"][0, p % 8] = ora.ids[p]
        for name, x in host.items():
            g.t[name].copy_(torch.from_numpy(x))
        g.st.cache_len = K
        for new in (3, 7, 4, 5, 1, 0, 5):
            attn = rng.random((U, K + 1)).astype(np.float32)
            state = {k: v.cpu().numpy() for k, v in g.t.items()}
            by_pos = []
            for u in range(U):
                d = {int(p): attn[u, r] for p, r in zip(state["pos"][u, :K], state["slot"][u, :K])}
                d[len(ora.ids)] = attn[u, state["next_slot"][u]]
                by_pos.append(d)
            ev = g.step(np.array([new], np.int32), attn)
            assert list(ev) == ora.step(new, by_pos)
            after = {k: v.cpu().numpy() for k, v in g.t.items()}
            for u, un in enumerate(ora.units):
                np.testing.assert_array_equal(after["pos"][u, :K], un.pos)
                np.testing.assert_array_equal(after["S"][u, :K], un.S)
                np.testing.assert_array_equal(after["tok"][u, :K], [ora.ids[p] for p in un.pos])
                for name, ref in (("A", un.A), ("P", un.P), ("V", un.V)):
                    np.testing.assert_array_equal(after[name][u, :K].view(np.uint32), np.array(ref, np.float32).view(np.uint32), name)
                assert sorted([*after["slot"][u, :K], after["next_slot"][u]]) == list(range(K + 1))
    finally:
        g.close()
