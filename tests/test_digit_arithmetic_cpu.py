"""The arithmetic of the digit products that host and device share, compiled for the host."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2305_09020_gb300 import _build

SRC = r"""
#define PF_TC_HELPERS_ONLY
#define PF_OZ_HELPERS_ONLY
#include "pf_oz.cuh"
#include <cstring>
extern "C" void quotients(int n, const double *x, const double *d, double *q) {
    for (int i = 0; i < n; ++i) q[i] = pf::oz_quot(x[i], pf::oz_recip(d[i]));
}
extern "C" void digits(int n, const double *x, const int *sh, int em, int *dig) {
    for (int i = 0; i < n; ++i) {
        unsigned long long u;
        std::memcpy(&u, &x[i], 8);
        const unsigned long long f = pf::oz_fixed(u, em - pf::oz_exp(u, sh[i]));
        for (int s = 0; s < pf::OZ_S; ++s) dig[i * pf::OZ_S + s] = (int)((f >> (8 * (pf::OZ_S - 1 - s))) & 0xFF) - 128;
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("digits")
    (d / "t.cu").write_text(SRC)
    subprocess.run([_build.nvcc(), _build.ARCH, "-std=c++17", "-O2", "-shared", "-Xcompiler", "-fPIC", "-Xcompiler",
                    "-ffp-contract=off", "-I", _build.CSRC, "-o", str(d / "t.so"), str(d / "t.cu")], check=True)
    return ctypes.CDLL(os.path.join(str(d), "t.so"))


def _p(a, t=ctypes.c_double):
    return a.ctypes.data_as(ctypes.POINTER(t))


def test_quotients_are_those_of_the_division_operator(lib):
    """Eigenvalue sums from 1e-140 to 1e140 and values from 1e-160 to 1e160: the same double in every case (the
    product with the rounded reciprocal differs in more than a tenth of them); a sum of 0 gives 0."""
    rng = np.random.default_rng(1)
    n = 400_000
    d = rng.uniform(1.0, 2.0, n) * 10.0 ** rng.uniform(-140, 140, n)
    x = rng.standard_normal(n) * 10.0 ** rng.uniform(-160, 160, n)
    d[:4] = [1.0, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -52, 0.0]
    q = np.empty(n)
    lib.quotients(n, _p(x), _p(d), _p(q))
    assert q[3] == 0.0
    keep = np.arange(n) != 3
    assert np.array_equal(q[keep], x[keep] / d[keep])
    assert np.mean(x[keep] * (1.0 / d[keep]) != x[keep] / d[keep]) > 0.1


def test_digits_hold_the_balanced_value(lib):
    """Exponents over the whole range, subnormals, zeros and shifts of both signs: the digits are those of the
    value in units of 2^(em - 1084), to half a unit, and within the bounds of the exact sums."""
    rng = np.random.default_rng(2)
    n = 20_000
    x = rng.standard_normal(n) * 2.0 ** rng.integers(-1060, 900, n)
    x[:6] = [0.0, -0.0, 5e-324, -1.5e-310, 2.2250738585072014e-308, -(2.0 - 2.0 ** -52) * 2.0 ** 899]
    sh = rng.integers(-900, 900, n).astype(np.int32)
    e = np.maximum((x.view(np.uint64) >> 52 & 0x7FF).astype(int), 1) + sh
    em = int(e[x != 0].max())
    for lo in (em, em - 300, em - 1500):               # rows whose largest exponent lies lower
        pick = e <= lo
        row, s = np.ascontiguousarray(x[pick]), np.ascontiguousarray(sh[pick])
        dig = np.empty((len(row), 8), dtype=np.int32)
        lib.digits(len(row), _p(row), _p(s, ctypes.c_int), lo, _p(dig, ctypes.c_int))
        assert dig.min() >= -128 and dig.max() <= 127 and np.abs(dig[:, 0]).max() <= 64
        for v, t, ds in zip(row[:2000], s, dig):
            X = sum(int(q) * 256 ** (7 - i) for i, q in enumerate(ds))
            m, p = np.frexp(v)                         # v = (m 2^53) 2^(p - 53), an integer and a power of two
            a, k = int(m * 2.0 ** 53), int(p) - 53 + int(t) - (lo - 1084)
            assert 2 * abs(X * 2 ** max(0, -k) - a * 2 ** max(0, k)) <= 2 ** max(0, -k)
