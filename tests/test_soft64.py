"""The FP64 filter's fixed-point functions (csrc/soft64.cuh), compiled for the host, against
extended precision.  The bounds are the stages' own: the tables and products carry 2^-60, the
normals' cosine and sine an absolute 2^-64 down to arguments of 2^-9, the exponential's argument
2^-57, and the result is rounded once to a double."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_12973_gb300", "csrc")
SOURCE = r"""
#include "soft64.cuh"
using namespace smc2;
extern "C" void normals(int n, const uint32_t* w, double* z) {
  for (int i = 0; i < n; ++i) s64_normal_pair(w[2 * i], w[2 * i + 1], g_soft64, z[2 * i], z[2 * i + 1]);
}
extern "C" void exps(int n, const double* x, uint64_t* m, int* k) {
  for (int i = 0; i < n; ++i) m[i] = s64_exp_q57(s64_q57(x[i]), g_soft64, k[i]);
}
extern "C" void log1p_minus(int n, const double* lam, const uint64_t* m, const int* e, double* g, int* ok) {
  for (int i = 0; i < n; ++i) {
    bool o;
    g[i] = s64_log1p_minus(lam[i], m[i], e[i], g_soft64, o);
    ok[i] = o;
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("soft64")
    src, so = str(d / "soft64.cpp"), str(d / "soft64.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    return C.CDLL(so)


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


def _ulp(x):
    return np.ldexp(np.longdouble(1), np.frexp(np.abs(x))[1] - 53)


@pytest.mark.parametrize("which", ["random", "first_near_one", "small_angle", "octant_edges"])
def test_normals(lib, which):
    rng = np.random.default_rng(1)
    w = rng.integers(0, 2 ** 32, (200000, 2), dtype=np.uint64).astype(np.uint32)
    k = np.arange(len(w), dtype=np.uint32)
    if which == "first_near_one":   # u_a up to 1 - 2^-24: -2 ln u_a down to 2^-23
        w[:, 0] = np.uint32(0xFFFFFFFF) - (k << np.uint32(6))
    elif which == "small_angle":
        w[:, 1] = k << np.uint32(9)
    elif which == "octant_edges":
        w[:, 1] = ((k & np.uint32(7)) << np.uint32(29)) + (((k >> np.uint32(3)) - np.uint32(12000)) << np.uint32(9))
    z = np.empty((len(w), 2))
    lib.normals(len(w), _p(np.ascontiguousarray(w)), _p(z))
    ua = np.longdouble(2 * (w[:, 0] >> 9).astype(np.int64) + 1) * np.longdouble(2) ** -24
    ub = np.longdouble(2 * (w[:, 1] >> 9).astype(np.int64) + 1) * np.longdouble(2) ** -24
    turn = np.rint(4 * ub)
    a = 2 * np.arctan2(np.longdouble(0), np.longdouble(-1)) * (ub - turn / 4)
    turn = turn.astype(np.int64) % 4
    # -ln u = ln(1 + (1 - u) / u), exact at u next to 1
    r = np.sqrt(2 * np.log1p((1 - ua) / ua))
    c, s = np.cos(a), np.sin(a)
    cos = np.choose(turn, [c, -s, -c, s])
    sin = np.choose(turn, [s, c, -s, -c])
    for got, ref in ((z[:, 0], r * cos), (z[:, 1], r * sin)):
        err = np.abs(got - ref) / _ulp(ref)
        assert err.max() < 1.5 and np.sqrt(np.mean(err ** 2)) < 0.35


def test_exponential(lib):
    rng = np.random.default_rng(2)
    x = np.concatenate([rng.uniform(-60, 60, 100000), -np.exp(rng.uniform(-40, 3.6, 100000)), [0.0, 2.0 ** -57, -37.0]])
    m, k = np.empty(len(x), np.uint64), np.empty(len(x), np.int32)
    lib.exps(len(x), _p(x), _p(m), _p(k))
    ref = np.exp(np.longdouble(x))
    got = np.ldexp(np.longdouble(m), k - 61)
    assert np.max(np.abs(got / ref - 1)) < 2.0 ** -56
    assert m[-3] == 2 ** 61 and k[-3] == 0   # e^0 is exactly one


@pytest.mark.parametrize("spread", [1e-6, 1e-3, 0.1, 0.9, 20.0])
def test_log1p_minus(lib, spread):
    rng = np.random.default_rng(3)
    n = 100000
    y = np.floor(np.exp(rng.uniform(0, 11, n)))
    lam = y * (np.exp(rng.uniform(-spread, spread, n)) if spread > 1 else 1 + rng.uniform(-spread, spread, n))
    inv = 1.0 / y
    e = (inv.view(np.uint64) >> 52).astype(np.int32) - 1023
    lo = (1 - np.longdouble(inv) * np.longdouble(y)) * np.longdouble(inv)
    m = (inv.view(np.uint64) << np.uint64(11)) | np.uint64(1 << 63)
    m = m + np.rint(np.ldexp(lo, 63 - e)).astype(np.int64).astype(np.uint64)
    g, ok = np.empty(n), np.empty(n, np.int32)
    lib.log1p_minus(n, _p(lam), _p(m), _p(e), _p(g), _p(ok))
    ratio = lam / y
    assert np.array_equal(ok.astype(bool), (np.floor(np.log2(ratio)) <= 5) & (ratio >= 2.0 ** -60))
    d = (np.longdouble(lam) - y) / np.longdouble(y)
    # log1p(d) - d without cancellation: d^2 (-1/2 + d/3 - ...) for small d
    small = np.abs(d) < 1e-3
    series = d * d * sum((-1) ** (j + 1) * d ** (j - 2) / j for j in range(2, 9))
    ref = np.where(small, series, np.where(ratio < 0.5, np.log(np.longdouble(lam) / np.longdouble(y)), np.log1p(d)) - d)
    sel = ok.astype(bool)
    near = (ratio > 0.7) & (ratio < 1.43)
    # near one: no more than the rounding of a double log1p(d), half an ulp of d
    tol = 2.0 ** -52 * np.abs(ref) + np.where(near, 2.0 ** -54 * np.abs(d) + 2.0 ** -76, 2.0 ** -54)
    assert np.all(np.abs(g - ref)[sel] <= tol[sel])
