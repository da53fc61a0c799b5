"""The arithmetic of the wide FFN that needs no GPU (csrc/ffn_wide_math.cuh), compiled for the host: the error of its GELU
against float64 and against the erf form of the math library, and the widths of its tiles."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
from scipy.special import erfc

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_08971_b200", "csrc")
SOURCE = r"""
#include "ffn_wide_math.cuh"
static float ulps(float x, int n) {
    for (; n > 0; --n) x = nextafterf(x, INFINITY);
    for (; n < 0; ++n) x = nextafterf(x, -INFINITY);
    return x;
}
extern "C" void gelu(const float* z, float* out, long n, int rcp_ulps, int ex2_ulps) {
    for (long i = 0; i < n; ++i)
        out[i] = gelu_two_part(z[i], [=](float x) { return ulps((float)(1.0 / (double)x), rcp_ulps); },
                               [=](float x) { return ulps((float)exp2((double)x), ex2_ulps); });
}
extern "C" int bn(int form, int R, int cols, int sm_count) { return wide_bn(form, R, cols, sm_count); }
extern "C" int bn_max(int form) { return wide_bn_max(form); }
extern "C" int second_one(int D, int k_c, long long rows, int token_ids, int n_lists) {
    return wide_second_one(D, k_c, rows, token_ids != 0, n_lists, 128, 148);
}
extern "C" int grid_cols(int cols) { return wide_grid_cols(cols); }
extern "C" void gelu_erf(const float* z, float* out, long n) {
    for (long i = 0; i < n; ++i) out[i] = 0.5f * z[i] * (1.f + erff(z[i] * 0.70710678f));
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    at = tmp_path_factory.mktemp("ffn_wide_math")
    (at / "host.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I" + CSRC, str(at / "host.cpp"), "-o",
                    str(at / "host.so"), "-lm"], check=True)
    return ctypes.CDLL(str(at / "host.so"))


def _call(f, z, *args):
    out = np.empty_like(z)
    at = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    f(at(z), at(out), ctypes.c_long(z.size), *args)
    return out.astype(np.float64)


def _exact(z):
    z = z.astype(np.float64)
    return 0.5 * z * erfc(-z * np.sqrt(0.5))


def test_gelu_error_is_no_larger_than_the_erf_form(lib):
    z = np.concatenate([np.linspace(-16, 16, 1000001), np.linspace(-1.3, 1.3, 500001)]).astype(np.float32)
    z = z[z != 0]
    worst = lambda g: float(np.max(np.abs(g - _exact(z)) / np.abs(z)))
    plain, erf_form = worst(_call(lib.gelu, z, 0, 0)), worst(_call(lib.gelu_erf, z))
    assert plain <= 1.0e-7 and plain <= erf_form, (plain, erf_form)
    # the device's 1/x is off by up to 1 ulp and its 2^x by up to 2: what they add at |z| >= 1 is Q(1) = 0.16 of
    # (1.2e-7 of 1/x, half of it in R, and 2.4e-7 of 2^x), 5e-8
    for ru in (-1, 1):
        for eu in (-2, 2):
            assert worst(_call(lib.gelu, z, ru, eu)) <= 1.5e-7
    rng = np.random.default_rng(0)
    for dev in (0.01, 0.03, 0.1, 0.3, 0.55, 1.0, 2.0, 3.0, 6.0):
        x = (rng.standard_normal(400000) * dev).astype(np.float32)
        rms = lambda g: float(np.sqrt(np.mean((g - _exact(x)) ** 2)))
        assert rms(_call(lib.gelu, x, 0, 0)) <= rms(_call(lib.gelu_erf, x)), dev
    # the tail keeps its digits: 2^-17 of the value is what the hidden buffer's head and remainder keep
    t = np.linspace(-12, -1, 300001).astype(np.float32)
    assert float(np.max(np.abs(_call(lib.gelu, t, 0, 0) / _exact(t) - 1))) <= 2.0 ** -17


def test_gelu_of_special_values(lib):
    inf, nan = float("inf"), float("nan")
    z = np.array([0.0, 1e-30, -1e-30, 20, -20, 1e19, -1e19, 2e38, -2e38, 3.4e38, -3.4e38, inf, -inf, nan], dtype=np.float32)
    g = _call(lib.gelu, z, 0, 0)
    finite = z[:-3].astype(np.float64)
    np.testing.assert_allclose(g[:-3], np.where(np.abs(finite) < 1, finite / 2, np.maximum(finite, 0)), rtol=1e-7, atol=0)
    assert np.isnan(g[-3:]).all()


FIRST, ONE, TWO = 0, 1, 2     # forms: GEMM 1, GEMM 2 with one and with two CTAs per SM
WIDEST = {FIRST: 160, ONE: 192, TWO: 128}


@pytest.mark.parametrize("form", [FIRST, ONE, TWO])
def test_every_column_has_a_block(lib, form):
    """The launch's blocks cover the columns at whichever width the device takes, and every width is taken."""
    taken = set()
    assert lib.bn_max(form) == WIDEST[form]
    for sm_count in (148, 132):
        for R in list(range(1, 129)):
            for cols in range(64, 1665, 64) if form == FIRST else range(64, 1025, 64):
                bn = lib.bn(form, R, cols, sm_count)
                assert 64 <= bn <= WIDEST[form] and bn % 32 == 0 and -(-cols // bn) <= lib.grid_cols(cols)
                taken.add(bn)
    assert taken == set(range(64, WIDEST[form] + 1, 32))


def test_second_form(lib):
    one = lambda D, k_c, rows, ids=0, lists=1: bool(lib.second_one(D, k_c, ctypes.c_longlong(rows), ids, lists))
    assert one(768, 1229, 37 * 128) and not one(768, 1229, 37 * 128 + 1)      # 148 tiles of 192 columns
    assert not one(768, 199, 128) and one(192, 200, 10 ** 9)                  # few K blocks; one column tile a row tile
    # several lists: two thirds of the rows of a call with masks, all of a call without
    assert one(768, 1229, 51 * 128, 1, 7) and not one(768, 1229, 53 * 128, 1, 7)
    assert one(768, 1229, 33 * 128, 0, 8) and not one(768, 1229, 34 * 128, 0, 8)


def test_gpu_shapes_take_every_width(lib):
    from tests.test_gpu_ffn_wide import WIDTHS
    taken, last = {FIRST: set(), ONE: set(), TWO: set()}, set()
    for D, k_c, tiles in WIDTHS:
        cols = (k_c + 63) // 64 * 64
        form = ONE if lib.second_one(D, k_c, ctypes.c_longlong(tiles * 128 - 37), 0, 1) else TWO
        a, b = lib.bn(FIRST, tiles, cols, 148), lib.bn(form, tiles, D, 148)
        taken[FIRST].add(a), taken[form].add(b), last.update((cols % a, D % b))
    assert taken == {form: set(range(64, WIDEST[form] + 1, 32)) for form in taken} and {32, 64, 128} <= last
