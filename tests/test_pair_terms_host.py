"""The binary64 form's fixed-point pair terms (csrc/expneg.cuh), compiled for the
host (the device code is the same source): the kernel exp(-d^2 / (2 h^2)) from
position images, the weight 2K / (r_i + r_j) and the 96-bit row sum, against
50-digit decimal arithmetic."""
import ctypes
import os
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_2204_03756_gb300 import build

SRC = """
#include "expneg.cuh"
using namespace mtpt;
extern "C" {
double kernel(int dim, const double* x, const double* y, double a, double psi) {
    double table[kExpTable];
    fill_exp_table(table);
    const KernelConsts c = kernel_consts(a, psi);
    uint64_t d2h = 0;
    for (int k = 0; k < dim; ++k) d2h += axis_square(x_image(x[k], c.x_shift), x_image(y[k], c.x_shift));
    return gauss_fixed(d2h, table, c);
}
double weight(double K, double ra, double rb) {
    const FixedWeight w = weight_fixed(K, ra, rb);
    return std::ldexp(double(w.q), w.x);
}
}
template <class Sum>
double sum_of(int n, const double* dm, const double* K, const double* ra, const double* rb) {
    Sum f;
    for (int k = 0; k < n; ++k) f.add(dm[k], weight_fixed(K[k], ra[k], rb[k]));
    return f.value();
}
extern "C" {
double flux_sum(int n, const double* dm, const double* K, const double* ra, const double* rb) {
    return sum_of<FluxSum64>(n, dm, K, ra, rb);
}
double adj_sum(int n, const double* dm, const double* K, const double* ra, const double* rb) {
    return sum_of<AdjSum64>(n, dm, K, ra, rb);
}
double row_sum(int n, const double* K) {
    RowSum r;
    for (int k = 0; k < n; ++k) r.add(unit_of(K[k]));
    return r.value();
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("terms")
    src, out = d / "terms.cpp", d / "terms.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-shared", "-fPIC", "-I", build.SRC_DIR,
                    "-o", str(out), str(src)], check=True)
    so = ctypes.CDLL(os.fspath(out))
    dp = ctypes.POINTER(ctypes.c_double)
    so.kernel.argtypes = [ctypes.c_int, dp, dp, ctypes.c_double, ctypes.c_double]
    so.weight.argtypes = [ctypes.c_double] * 3
    so.row_sum.argtypes = [ctypes.c_int, dp]
    so.flux_sum.argtypes = so.adj_sum.argtypes = [ctypes.c_int, dp, dp, dp, dp]
    for f in (so.kernel, so.weight, so.row_sum, so.flux_sum, so.adj_sum):
        f.restype = ctypes.c_double
    getcontext().prec = 50
    return so


def _ptr(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


@pytest.mark.parametrize("lam,h2,side", [(3.0, 0.1, 100.0), (3.0, 0.1, 2000.0), (3.0, 1e-30, 1e-9),
                                         (3.0, 7.0, 1e15), (0.001, 0.1, 10.0), (20.0, 0.05, 126.0)])
@pytest.mark.parametrize("dim", [1, 2, 3])
def test_kernel_against_decimal(lib, lam, h2, side, dim):
    rng = np.random.default_rng(dim)
    psi, a = lam * np.sqrt(2.0 * h2), 1.0 / (2.0 * h2)
    # |T's error| <= 3 + 6 d units of 2^-60 (psi^2) in d2 and the constant's
    # 2^-63: a relative error of K of lam^2 (3 + 6 d) 2^-60 at most, plus the
    # rounding of T (4 units of at most lam^2 2^-57) and of the table, the series
    # and their product (2^-53 each)
    bound = 3 * 2.0 ** -53 + lam ** 2 * ((3 + 6 * dim) * 2.0 ** -60 + 4 * 2.0 ** -57) + 2.0 ** -58
    for it in range(300):
        x = rng.uniform(-side, side, dim) * (1e-3 if it % 3 == 0 else 1.0)
        y = x + rng.uniform(-1.0, 1.0, dim) * psi / np.sqrt(dim) * (it % 7 != 0)
        d2 = sum((Decimal(float(u)) - Decimal(float(v))) ** 2 for u, v in zip(x, y))
        if d2 > Decimal(psi) ** 2:
            continue
        want = (-Decimal(a) * d2).exp()
        got = lib.kernel(dim, _ptr(x), _ptr(y), a, psi)
        assert lib.kernel(dim, _ptr(y), _ptr(x), a, psi) == got
        assert abs(Decimal(got) - want) <= Decimal(bound) * want
        if d2 == 0:
            assert got == 1.0


def test_weight_against_decimal(lib):
    rng = np.random.default_rng(4)
    for it in range(4000):
        K = float(np.exp(-rng.uniform(0.0, 9.0 if it % 2 else 400.0)))
        ra = 1.0 + (rng.uniform(0.0, 60.0) if it % 5 else 0.0)
        rb = 1.0 + rng.uniform(0.0, 2.0 ** 30 if it % 3 == 0 else 2.0)
        want = 2 * Decimal(K) / (Decimal(ra) + Decimal(rb))
        got = lib.weight(K, ra, rb)
        assert got == lib.weight(K, rb, ra)
        assert abs(Decimal(got) - want) <= Decimal(2.0 ** -53 + 2.0 ** -54) * want
    assert lib.weight(1.0, 1.0, 1.0) == 1.0


@pytest.mark.parametrize("n", [0, 1, 2, 3, 4, 7, 8, 63, 64, 1000, 5000])
def test_row_sum_against_decimal(lib, n):
    """1 + sum K: every term to 2^-62, one rounding at the end."""
    rng = np.random.default_rng(n)
    K = np.exp(-rng.uniform(0.0, 9.0, n))
    if n > 2:
        K[:2] = (1.0, 2.0 ** -70)
    want = Decimal(1) + sum((Decimal(float(k)) for k in K), Decimal(0))
    got = lib.row_sum(n, _ptr(K))
    assert abs(Decimal(got) - want) <= Decimal(2.0 ** -53) * want + n * Decimal(2) ** -62


@pytest.mark.parametrize("n", [0, 1, 2, 5, 31, 33, 64, 2000])
@pytest.mark.parametrize("spread", [0, 40, 1000])
def test_flux_sum_against_decimal(lib, n, spread):
    """sum W dm over masses of one size and of sizes 2^+-spread apart: every term
    to 2^-52 of the largest, and the sum rounded once; of the opposite differences,
    exactly the opposite sum."""
    rng = np.random.default_rng(n + spread)
    dm = rng.uniform(-1.0, 1.0, n) * 2.0 ** rng.integers(-spread, 1, n)
    if n > 3:
        dm[:2] = (0.0, -0.0)
    K, ra, rb = np.exp(-rng.uniform(0.0, 9.0, n)), 1.0 + rng.uniform(0, 9, n), 1.0 + rng.uniform(0, 9, n)
    terms = [2 * Decimal(float(k)) / (Decimal(float(a)) + Decimal(float(b))) * Decimal(float(m))
             for k, a, b, m in zip(K, ra, rb, dm)]
    want = sum(terms, Decimal(0))
    big = max([abs(t) for t in terms], default=Decimal(0))
    for f in (lib.adj_sum, lib.flux_sum):
        got = f(n, _ptr(dm), _ptr(K), _ptr(ra), _ptr(rb))
        assert abs(Decimal(got) - want) <= Decimal(2.0 ** -52) * n * big + Decimal(2.0 ** -53) * abs(want)
    assert lib.flux_sum(n, _ptr(-dm), _ptr(K), _ptr(ra), _ptr(rb)) == -got


@pytest.mark.parametrize("n", [7, 8, 9, 100, 5000])
@pytest.mark.parametrize("m", [1.0, -1.0, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -52, 1e-300])
def test_flux_sum_of_many_like_terms(lib, n, m):
    """Terms of one sign, which raise the unit as the sum grows: less than two units
    of 2^-57 of the sum for each, and the sum rounded once."""
    K, r = np.full(n, 0.7310585786300049), np.full(n, 3.3)
    dm = np.full(n, m)
    want = n * Decimal(m) * 2 * Decimal(K[0]) / (2 * Decimal(r[0]))
    # (the weight and the product are each within 2^-54 too)
    bound = Decimal(2 * n * 2.0 ** -57 + 3 * 2.0 ** -54 + 2.0 ** -53) * abs(want)
    for f in (lib.adj_sum, lib.flux_sum):
        got = f(n, _ptr(dm), _ptr(K), _ptr(r), _ptr(r))
        assert abs(Decimal(got) - want) <= bound
    assert lib.flux_sum(n, _ptr(-dm), _ptr(K), _ptr(r), _ptr(r)) == -got


def test_flux_sum_of_differences_that_are_not_finite(lib):
    one = np.ones(3)
    for dm, want in ((np.array([1.0, np.inf, 2.0]), np.inf), (np.array([-np.inf, 5.0, 1.0]), -np.inf),
                     (np.array([np.inf, -np.inf, 1.0]), np.nan), (np.array([1.0, np.nan, 1.0]), np.nan)):
        got = lib.flux_sum(3, _ptr(dm), _ptr(one), _ptr(one), _ptr(one))
        assert got == want or (np.isnan(want) and np.isnan(got))
    big = np.array([1.5e308, -1.5e308, 1e300])
    assert np.isfinite(lib.flux_sum(3, _ptr(big), _ptr(one), _ptr(one), _ptr(one)))
