"""Block fixed point (csrc/swdg_fixed.cuh) on the host, against exact sums.

Tolerance, in units of 2^-60 of the result's bound 2^(eb - 1022 + t): half a
unit from the values' conversions (their errors weighted by a table row of sum
at most 2^t), half a unit per term from the table's digits, a quarter per term
from the digit product left out, half from the final shift; then the conversion
back rounds at 2^-53 of the result.
"""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2505_18743_gb300", "csrc")
SRC = r"""
#include "swdg_fixed.cuh"
#include <cmath>
using namespace swdg;
extern "C" int fx_dot(const double* T, const double* v, int n, double* out) {
    double s = 0.0;
    unsigned m = 0;
    for (int i = 0; i < n; ++i) { s += std::fabs(T[i]); m = fx::mag(v[i]) > m ? fx::mag(v[i]) : m; }
    int t = -64;
    while (std::ldexp(1.0, t) < s) ++t;
    const int e = fx::block_exp(m);
    fx::Acc a;
    for (int i = 0; i < n; ++i)
        a.mac(fx::split(std::llrint(std::ldexp(T[i], fx::FB - t))), fx::split(fx::from_double(v[i], e)));
    *out = fx::to_double(a.get(), e + t);
    return e + t;
}
extern "C" void fx_float(const float* v, int n, double* out, float* back) {
    unsigned m = 0;
    for (int i = 0; i < n; ++i) { const unsigned b = fx::fbits(v[i]) & 0x7fffffffu; m = b > m ? b : m; }
    const int e = fx::block_exp_f(m);
    for (int i = 0; i < n; ++i) {
        const long long X = fx::from_float(v[i], e);
        out[i] = fx::to_double(X, e);
        back[i] = fx::to_float(X, e);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cu").write_text(SRC)
    so = d / "fx.so"
    subprocess.run([nvcc, "-shared", "-Xcompiler", "-fPIC", "-std=c++17", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I", CSRC, "-o", str(so), str(d / "fx.cu")],
                   check=True, capture_output=True)
    return ctypes.CDLL(str(so))


def _dot(lib, T, v):
    out = ctypes.c_double()
    p = ctypes.POINTER(ctypes.c_double)
    T, v = np.ascontiguousarray(T, float), np.ascontiguousarray(v, float)
    e = lib.fx_dot(T.ctypes.data_as(p), v.ctypes.data_as(p), len(T), ctypes.byref(out))
    return out.value, e


@pytest.mark.parametrize("n", [1, 2, 5, 13])
@pytest.mark.parametrize("spread", [0, 12, 300])
def test_contraction_error_is_within_its_bound(lib, n, spread):
    rng = np.random.default_rng(100 * n + spread)
    for _ in range(300):
        T = rng.standard_normal(n) * 2.0 ** rng.integers(-3, 4)
        v = rng.standard_normal(n) * 2.0 ** (rng.integers(-spread, spread + 1, n) if spread else 0)
        v[rng.random(n) < 0.1] = 0.0
        got, e = _dot(lib, T, v)
        exact = sum((Fraction(a) * Fraction(b) for a, b in zip(T, v)), Fraction(0))
        unit = Fraction(2) ** (e - 1022 - 60)
        bound = unit * Fraction(1 + n * 3, 1) + abs(exact) * Fraction(1, 2 ** 52)
        assert abs(Fraction(got) - exact) <= bound


def test_infinities_nans_and_vanishing_blocks(lib):
    for bad in (np.inf, -np.inf, np.nan):
        assert np.isnan(_dot(lib, [0.5, 0.25], [1.0, bad])[0])
    assert _dot(lib, [0.5, 0.25], [0.0, -0.0])[0] == 0.0
    assert _dot(lib, [0.5, 0.25], [5e-324, 1e-307])[0] == 0.0  # values below 2^-1018
    assert _dot(lib, [1.0], [np.finfo(float).max])[0] == pytest.approx(np.finfo(float).max, rel=2e-16)


def test_fp32_values_are_exact_within_36_places_of_the_largest(lib):
    rng = np.random.default_rng(4)
    v = (rng.standard_normal(64) * 2.0 ** rng.integers(-35, 1, 64)).astype(np.float32)
    v[:3] = 4.0, 0.0, -2.0 ** -30
    out, back = np.empty(64), np.empty(64, np.float32)
    lib.fx_float(v.ctypes.data_as(ctypes.c_void_p), 64, out.ctypes.data_as(ctypes.c_void_p),
                 back.ctypes.data_as(ctypes.c_void_p))
    big = np.abs(v) >= 2.0 ** -34
    assert np.array_equal(out[big], v[big].astype(float)) and np.array_equal(back[big], v[big])
    assert np.abs(out - v).max() <= 2.0 ** -58
