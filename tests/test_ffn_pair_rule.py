"""The GPU tests that compare CTA pairs of the fused FFN with single CTAs reach both forms: the rule of csrc/ffn_pair_rule.cuh,
compiled for the host, at their shapes on 148 SMs."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_08971_b200", "csrc")
SOURCE = r"""
#include "ffn_pair_rule.cuh"
extern "C" int takes_pairs(int token_ids, int n_lists, int k_c, long long max_tiles, int sm_count) {
    return ffn_takes_pairs(token_ids != 0, n_lists, k_c, max_tiles, sm_count);
}
"""


@pytest.fixture(scope="module")
def takes_pairs(tmp_path_factory):
    at = tmp_path_factory.mktemp("ffn_pair_rule")
    (at / "host.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(at / "host.cpp"), "-o", str(at / "host.so")],
                   check=True)
    f = ctypes.CDLL(str(at / "host.so")).takes_pairs
    return lambda ids, lists, k_c, rows: bool(f(int(ids), lists, k_c, ctypes.c_longlong(-(-rows // 128) + lists), 148))


def test_masked_calls(takes_pairs):
    from tests.test_gpu_ffn_tmem import PAIR_STEP, PAIR_T, PAIRS
    assert {d for k, _, _, d in PAIRS if k > 128} == {"bf16", "f16"}
    for k_c, lists, B, _ in PAIRS:
        assert takes_pairs(True, lists, k_c, B * PAIR_T) == (k_c > 128), (k_c, lists, B)
        assert not takes_pairs(True, lists, k_c, PAIR_STEP * PAIR_T)


def test_sparse_moe_calls(takes_pairs):
    from tests.test_gpu_moe import PAIR_STEP, PAIR_TOP_K, PAIRS
    for E, k_c, N in PAIRS:
        assert takes_pairs(False, E, k_c, N * PAIR_TOP_K), (E, k_c, N)
        assert not takes_pairs(False, E, k_c, PAIR_STEP * PAIR_TOP_K)


def test_never(takes_pairs):
    for ids in (False, True):
        assert not takes_pairs(ids, 1, 128, 10 ** 8)       # one chunk of channels
        assert not takes_pairs(ids, 65, 512, 10 ** 8)      # every thread adds up the lists
