"""Block fixed point (csrc/swdg_fixed.cuh) on the host at the limits of its format:
digit pairs and renormalised blocks at 2^60, and contractions whose values and
table rows both reach their bounds.

Tolerance of a contraction of n terms, in units of 2^-60 of the result's bound: half a
unit from the values' conversions (weighted by a table row of sum at most 2^t),
half a unit a term from the table's digits, a quarter a term from the digit product
left out, half from the final shift: 1 + 3 n / 4.
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
extern "C" long long fx_split_join(long long X) { return fx::join(fx::split(X)); }
extern "C" int fx_headroom(const long long* X, int n) {
    unsigned m = 0;
    for (int i = 0; i < n; ++i) m = fx::high(X[i]) > m ? fx::high(X[i]) : m;
    return fx::headroom(m);
}
// n terms against a table of scale 2^t: the sum as an integer at exponent e + t
extern "C" long long fx_sum(const double* T, const double* v, int n, int t, int* e) {
    unsigned m = 0;
    for (int i = 0; i < n; ++i) m = fx::mag(v[i]) > m ? fx::mag(v[i]) : m;
    *e = fx::block_exp(m);
    fx::Acc a;
    for (int i = 0; i < n; ++i)
        a.mac(fx::split(std::llrint(std::ldexp(T[i], fx::FB - t))), fx::split(fx::from_double(v[i], *e)));
    return a.get();
}
extern "C" long long fx_product(long long a, long long b) { return fx::product(fx::split(a), fx::split(b)); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("fxl")
    (d / "fx.cu").write_text(SRC)
    so = d / "fx.so"
    subprocess.run([nvcc, "-shared", "-Xcompiler", "-fPIC", "-std=c++17", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I", CSRC, "-o", str(so), str(d / "fx.cu")],
                   check=True, capture_output=True)
    lib = ctypes.CDLL(str(so))
    lib.fx_split_join.restype = lib.fx_sum.restype = lib.fx_product.restype = ctypes.c_longlong
    lib.fx_split_join.argtypes = [ctypes.c_longlong]
    lib.fx_product.argtypes = [ctypes.c_longlong] * 2
    return lib


@pytest.mark.parametrize("k", list(range(1, 61)))
def test_renormalised_blocks_keep_their_digits(lib, k):
    for X in (2 ** k, 2 ** k - 1, 2 ** k - 2, -2 ** k, 1 - 2 ** k, 2 - 2 ** k):
        s = lib.fx_headroom((ctypes.c_longlong * 2)(X, 0), 2)
        Y = X << s
        assert s >= 0 and abs(Y) <= 2 ** 60
        assert lib.fx_split_join(Y) == Y
        # the largest place that is sure from the high word is used
        assert abs(X) < 2 ** 32 or abs(X) == 2 ** 60 or abs(Y) >= 2 ** 59
        # a product with the largest value of another block
        for Z in (2 ** 60 - 1, -2 ** 60):
            assert abs(lib.fx_product(Y, Z) - Fraction(Y * Z, 2 ** 60)) <= 1


@pytest.mark.parametrize("n", [1, 2, 5, 13])
def test_contractions_at_their_bounds(lib, n):
    rng = np.random.default_rng(n)
    P = ctypes.POINTER(ctypes.c_double)
    for case in range(200):
        w = rng.integers(1, 1000, n)
        T = w / 1024.0
        T[-1] += 2.0 ** np.ceil(np.log2(T.sum())) - T.sum()  # the row's sum is 2^t exactly
        t = int(np.log2(T.sum()))
        assert T.sum() == 2.0 ** t
        sg = rng.choice([-1.0, 1.0], n)
        v = sg * np.nextafter(2.0, 0.0) * (1.0 if case % 2 else 1.0 - rng.random(n) * 2.0 ** -20)
        T = T * (sg if case % 4 < 2 else 1.0)  # every term of one sign, or mixed
        e = ctypes.c_int()
        X = lib.fx_sum(np.ascontiguousarray(T).ctypes.data_as(P), np.ascontiguousarray(v).ctypes.data_as(P),
                       n, t, ctypes.byref(e))
        exact = sum((Fraction(a) * Fraction(b) for a, b in zip(T, v)), Fraction(0))
        unit = Fraction(2) ** (e.value + t - 1022 - 60)
        assert abs(X - exact / unit) <= 1 + Fraction(3 * n, 4)
        assert abs(X) <= 2 ** 60 + 1 + n and lib.fx_split_join(X) == X
