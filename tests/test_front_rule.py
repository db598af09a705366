"""How many blocks share a sequence or a unit, and that a device which does not hold their clusters at once is given something else:
the rules are host code, compiled here by themselves."""
import ctypes
import os
import subprocess

import pytest

import paper_2604_11288_b200 as ta

INCLUDE = os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")
SOURCE = r"""
#include "ta_front_rule.h"
#include "ta_internal.cuh"
extern "C" int helped(int K, int units, int held) { return ta_select_helped(K, units, held); }
extern "C" int blocks(int n, int batch, int sms, int score_units, int selects, const int* fits) {
  return ta_front_blocks(n, batch, sms, score_units, selects != 0, [&](int cl) { return cl == 16 ? fits[3] : cl == 8 ? fits[2] : cl == 4 ? fits[1] : fits[0]; });
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text(SOURCE)
    csrc = os.path.join(os.path.dirname(ta.__file__), "csrc")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-fPIC", "-shared", "-I", csrc, "-I", INCLUDE,
                    "-I", os.path.join(os.path.dirname(os.path.dirname(ta.__file__)), "include"), str(d / "rule.cpp"), "-o",
                    str(d / "rule.so")], check=True)
    lib = ctypes.CDLL(str(d / "rule.so"))

    def blocks(n, batch, fits, score_units=0, selects=True, sms=148):
        return lib.blocks(n, batch, sms, score_units, int(selects), (ctypes.c_int * 4)(*fits))
    blocks.helped = lib.helped
    return blocks


B200 = (74, 33, 15, 7)  # clusters of 2, 4, 8, 16 blocks
SIZES = [1, 12288, 12289, 16384, 16385, 32768, 32769, 65536, 65537, 131072, 131073, 262144, 262145]


@pytest.mark.parametrize("score_units", [0, 1, 12, 256])
@pytest.mark.parametrize("fits", [B200, (0, 0, 0, 0), (74, 0, 0, 0), (74, 33, 15, 0), (0, 0, 3, 1), (9, 4, 0, 0)])
def test_only_sizes_that_hold_the_sequence_and_that_the_device_holds(rule, fits, score_units):
    for n in SIZES:
        for batch in (1, 2, 7, 8, 15, 16, 33, 34, 74, 75, 1000):
            cl = rule(n, batch, fits, score_units)
            able = [c for c, f in zip((1, 2, 4, 8, 16), (1,) + fits) if c * 16384 >= n and f > 0]
            assert cl in able or (cl == 0 and (not able or n > 131072)), (n, batch, cl)
            if n <= 12288:
                assert cl == 1


def test_all_clusters_at_once_where_they_fit(rule):
    assert [rule(20000, b, B200) for b in (15, 16, 33, 34, 74, 75)] == [8, 4, 4, 2, 2, 2]
    assert rule(200000, 3, (74, 33, 15, 0)) == 0
    assert rule(20000, 20, (0, 0, 0, 0)) == 0


def test_helping_blocks_only_where_all_clusters_run_at_once(rule):
    assert [rule.helped(512, u, 33) for u in (1, 33, 34, 35)] == [1, 1, 0, 0]
    assert rule.helped(511, 8, 33) == 0 and rule.helped(4096, 1, 0) == 0


def test_sequences_that_need_the_largest_clusters(rule):
    # one kernel per step where a last round would hold one cluster, and where a score kernel of few units finds no room beside them
    assert [rule(200000, b, B200) for b in (1, 7, 8, 9, 14, 15, 16, 22, 100)] == [16, 16, 0, 16, 16, 0, 16, 16, 16]
    assert [rule(200000, b, B200, 8 * b) for b in (1, 2, 3, 4, 5, 8, 15)] == [16, 16, 0, 16, 16, 16, 16]
    assert [rule(200000, b, B200, 2 * b) for b in (2, 3, 4, 5, 7)] == [16, 16, 0, 16, 16]
    assert [rule(200000, 4, B200, u) for u in (4, 8, 12, 16)] == [16, 0, 0, 16]
    assert [rule(200000, b, (0, 0, 0, 1)) for b in (1, 2, 3)] == [16, 16, 16]


def test_blocks_beside_a_score_kernel_and_without(rule):
    assert [rule(n, 4, B200) for n in (12288, 12289, 32768, 32769)] == [1, 8, 8, 16]
    assert [rule(n, 4, B200, 0, False) for n in (12288, 12289, 32769)] == [1, 16, 16]
    assert [rule(n, 8, B200, 0, False) for n in (12289, 32768, 32769)] == [8, 8, 8]
    assert [rule(n, 4, B200, 32, False) for n in (16384, 16385, 32768, 32769, 131072)] == [1, 8, 8, 16, 16]
