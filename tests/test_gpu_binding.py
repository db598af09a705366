"""The frequent calls give the same results through the native marshalling module and through ctypes."""
import numpy as np
import pytest
import torch

import paper_2604_11288_b200 as ta
import ta_workloads as tw
from ta_testlib import Gpu, oracle_policy

pytestmark = pytest.mark.gpu


def _run_all():
    w = tw.config1(n=1024 + 77, Hq=8, Hkv=2)
    Q, Kc, Vc = (t.cuda() for t in tw.make_qkv(w, [0]))
    g = Gpu(w, oracle_policy(16, "THEOREM", W=w.W), 16, 1)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    out = []
    try:
        out += g.compress(Q, Kc, Vc)
        score = torch.rand((1, w.Hkv, w.total), generator=gen, device="cuda")
        out += g.compress_scores(score, None, Kc, Vc)
        lse = torch.rand((1, w.B, w.Hq, w.W), generator=gen, device="cuda") + 5.0
        idx, cnt = torch.zeros_like(out[0]), torch.zeros_like(out[1])
        ko, vo = torch.zeros_like(out[2]), torch.zeros_like(out[3])
        ta.ta_compress_lse(g.ctx, g.pats, g.p, g.batch, w.Hq, w.Hkv, w.d, 16, g.ids, ta.view(Q), ta.view(Kc), ta.view(Vc), lse,
                           0, ko, vo, idx, cnt, g.stream)
        out += [idx, cnt, ko, vo]
        emb = torch.randn((w.total, 64), generator=gen, dtype=torch.bfloat16, device="cuda")
        concepts = torch.randn((5, 64), generator=gen, dtype=torch.bfloat16, device="cuda")
        conf = torch.zeros(w.total, device="cuda")
        ta.ta_detect_embedding(g.ctx, w.total, emb, 64, 64, concepts, 5, conf, g.stream)
        out += [conf, *g.sponsor_mask_conf(conf, 0.2, 15.0, 6, True)]
        assert g.poll() == ta.TA_OK
    finally:
        g.close()
    return [t.cpu() for t in out]


def test_results_do_not_depend_on_the_marshalling(monkeypatch):
    a = _run_all()
    assert type(ta.binding._call).__name__ == "module"
    monkeypatch.setattr(ta.binding, "_call", ta.binding._CtypesCalls(ta.binding.lib()))
    b = _run_all()
    for x, y in zip(a, b, strict=True):
        np.testing.assert_array_equal(x.view(torch.uint8).numpy(), y.view(torch.uint8).numpy())
