"""CPU-side checks of the CUDA library: it builds for sm_100a, loads without a GPU, exports every entry point that
include/ta.h declares, and its pure-host helpers behave. No kernel is launched here."""
import ctypes as C
import os
import re
import subprocess

import pytest

import paper_2604_11288_b200 as ta
from paper_2604_11288_b200 import build as ta_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    ta_build.build()
    return ta.binding.lib()


def _declared():
    text = open(os.path.join(ROOT, "include", "ta.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(ta_[a-z_0-9]+)\s*\(", text)))


def test_exports_every_declared_symbol(lib):
    names = _declared()
    assert {"ta_sponsor_mask", "ta_score", "ta_select_topk", "ta_compact_kv", "ta_compress"} <= set(names)
    for n in names:
        assert hasattr(lib, n), n


def test_policy_presets(lib):
    p = ta.ta_policy_default(ta.TA_PRESET_THEOREM, 16)
    assert (p.n_sink, p.n_recent, p.k_protected) == (1, 4, -1)
    assert (round(p.alpha, 3), round(p.beta, 3), round(p.gamma, 3), round(p.delta, 3), round(p.lambda_, 3)) == \
        (1.0, 0.5, 0.3, 0.2, 0.1)
    assert round(p.voucher_decay, 3) == 0.8 and round(p.budget_decay, 3) == 0.9
    p = ta.ta_policy_default(ta.TA_PRESET_SEC33, 16)
    assert (p.n_sink, p.n_recent, p.k_protected) == (1, 2, 4)  # K=16 -> 12 + 4
    p = ta.ta_policy_default(ta.TA_PRESET_AUDIT, 16)
    assert (p.n_sink, p.n_recent, p.k_protected) == (4, 6, 6)
    with pytest.raises(ta.TAError):
        ta.ta_policy_default(9, 16)


def test_scratch_size_and_validation(lib):
    p = ta.ta_policy_default(0, 16)
    b = ta.make_batch(32, 1, 4096, 4096, 4096)
    scored = ta.ta_scratch_bytes(b, 32, 8, 128, 16, p)
    assert scored >= 32 * 8 * 4096 * 4  # the fused utilities
    p.mode = ta.TA_MODE_FAST
    assert ta.ta_scratch_bytes(b, 32, 8, 128, 16, p) < scored
    bad = ta.make_batch(1, 2, 100, 100, 150)  # total != B * n
    with pytest.raises(ta.TAError) as e:
        ta.ta_scratch_bytes(bad, 32, 8, 128, 16, p)
    assert e.value.status == ta.TA_ERR_INVALID_ARG
    assert "invalid" in ta.status_string(ta.TA_ERR_INVALID_ARG)


def test_no_device_is_an_error_not_a_crash(lib):
    import torch
    if torch.cuda.is_available():
        pytest.skip("a device is present")
    h = C.c_void_p()
    assert lib.ta_ctx_create(0, 1024, C.byref(h)) != ta.TA_OK
    assert not h.value


def test_missing_library_fails_loudly(monkeypatch, tmp_path):
    monkeypatch.setattr(ta.binding, "_lib", None)
    monkeypatch.setattr(ta.binding, "LIB_PATH", str(tmp_path / "libta.so"))
    with pytest.raises(FileNotFoundError):
        ta.binding.lib()


def test_score_kernel_keeps_its_values_in_registers(tmp_path):
    # setmaxnreg leaves the statistics warps 56 registers; what does not fit goes to local memory on the path between the
    # two passes. A spilled scalar or two outside the loops is tolerated, an array is not.
    csrc = os.path.join(ROOT, "paper_2604_11288_b200", "csrc")
    out = subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a",
                          "-O3", "-lineinfo", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", csrc, "-Xptxas", "-v",
                          "-c", os.path.join(csrc, "ta_score.cu"), "-o", str(tmp_path / "score.o")],
                         check=True, capture_output=True, text=True).stderr
    spills = dict(re.findall(r"Compiling entry function '(\S*ta_score_kernel\S*)'.*?(\d+) bytes spill stores", out, re.S))
    assert len(spills) == 6
    assert max(int(n) for n in spills.values()) <= 8, spills


@pytest.fixture
def ctypes_calls(lib, monkeypatch, tmp_path):
    """The binding as it loads where the native module is missing."""
    monkeypatch.setattr(ta.binding, "_lib", None)
    monkeypatch.setattr(ta.binding, "_call", None)
    monkeypatch.setattr(ta.binding, "CALL_PATH", str(tmp_path / "_ta_call.so"))
    ta.binding.lib()
    return ta.binding._call


def _refused(calls):
    """Status of every call of the native module without a context (nothing reaches a device)."""
    p, b, v, st = ta.ta_policy_default(0, 16), ta.make_batch(1, 1, 64, 64, 64), ta.ta_bf16_view(), ta.ta_stream()
    return [calls.ta_compress(None, None, p, b, 8, 2, 128, 16, None, v, v, v, 0, None, None, None, None, None),
            calls.ta_compress_lse(None, None, p, b, 8, 2, 128, 16, None, v, v, v, None, 0, None, None, None, None, None),
            calls.ta_compress_scores(None, None, p, b, 2, 128, 16, None, None, None, v, v, 0, None, None, None, None, None),
            calls.ta_stream_step(None, None, p, st, None, None, None, None),
            calls.ta_detect_embedding(None, 64, None, 2048, 2048, None, 8, None, None),
            calls.ta_sponsor_mask_conf(None, p, b, None, None, 0.5, 15.0, 6, 0, None, None, None, None)]


def test_library_loads_without_the_native_module(lib, ctypes_calls, monkeypatch):
    import torch
    assert type(ctypes_calls).__name__ == "_CtypesCalls"
    with pytest.raises(ta.TAError):
        ta.ta_stream_step(None, None, ta.ta_policy_default(0, 16), ta.ta_stream(), None, None, None)
    monkeypatch.undo()
    native = ta.binding._native()
    assert type(native).__name__ == "module"
    assert _refused(ctypes_calls) == _refused(native) == [ta.TA_ERR_INVALID_ARG] * 6
    for t, ragged in ((torch.zeros(2, 3, 4, 8, 128, dtype=torch.bfloat16)[:, :, 1:], False),
                      (torch.zeros(2, 4, 9, 128, dtype=torch.bfloat16), True), (None, False)):
        assert bytes(ctypes_calls.view(t, ragged)) == bytes(native.view(t, ragged))
    for bad, ragged in ((torch.zeros(2, 3, 8, 128), False), (torch.zeros(1, 2, 3, 128, 8).transpose(3, 4), False),
                        (torch.zeros(2, 3, 4, 8, 128), True)):
        for c in (ctypes_calls, native):
            with pytest.raises(AssertionError):
                c.view(bad, ragged)


def test_native_module_is_of_this_python(lib):
    import sysconfig
    assert ta.binding.CALL_PATH == ta_build.CALL_PATH
    assert ta.binding.CALL_PATH.endswith(sysconfig.get_config_var("EXT_SUFFIX"))


def test_build_without_a_compiler_for_the_module(lib, monkeypatch, tmp_path, capfd):
    monkeypatch.setattr(ta_build, "CALL_PATH", str(tmp_path / "_ta_call.so"))
    monkeypatch.setenv("CXX", str(tmp_path / "no_such_compiler"))
    assert ta_build.build() == ta_build.LIB_PATH
    assert not os.path.exists(ta_build.CALL_PATH) and "ctypes" in capfd.readouterr().err
