"""The FP64 kernels' reciprocal, weight and deformation determinant (`qrcp`, `transform64`, `weight64`, `det_deform` in
csrc/qmc_dev.cuh), and the default launch shape, checked on the host without a GPU.

The device source is cut out as written and compiled with g++; the 20-bit reciprocal approximation of the hardware is
replaced by a value with a relative error of 2^-20, the worst it is used for."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

import workloads as W
from paper_1508_02512_gb300 import _native as N
from paper_1508_02512_gb300 import api
from paper_1508_02512_gb300 import tables as T

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WORK = os.path.join(ROOT, "tests", "_gen_build")
SRC = os.path.join(ROOT, "paper_1508_02512_gb300", "csrc", "qmc_dev.cuh")

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
using std::fma;
#define DEV static inline
#define __shared__
struct cd { double x, y; };
DEV cd mk(double x, double y) { return cd{x, y}; }
DEV cd cmul(cd a, cd b) { return cd{fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x)}; }
static inline long long __double_as_longlong(double d) { long long b; std::memcpy(&b, &d, 8); return b; }
static inline int __double2hiint(double d) { return (int)(__double_as_longlong(d) >> 32); }
static inline double __drcp_rn(double x) { return 1.0 / x; }
DEV double rcp_seed(double x) { return (1.0 + (x > 0 ? 1 : -1) * 9.5367431640625e-7) / x; }
"""

TAIL = r"""
extern "C" void h_qrcp(const double *x, double *y, long n) { for (long i = 0; i < n; ++i) y[i] = qrcp(x[i]); }
extern "C" void h_transform(int r, const double *x, double *t, double *tm, double *w, long n) {
    for (long i = 0; i < n; ++i) { double xy; transform64(r, x[i], t[i], tm[i], xy); w[i] = weight64<1>(r, xy); }
}
template <int S> static void det_s(const double *T, const double *a, const double *h, double lam, unsigned Y, double *o) {
    double t[S], d[S];
    for (int j = 0; j < S; ++j) { t[j] = T[j]; d[j] = a[j]; }
    const cd v = det_deform<S>(t, d, h, lam, Y);
    o[0] = v.x;
    o[1] = v.y;
}
extern "C" void h_det(int S, const double *T, const double *a, const double *h, double lam, unsigned Y, double *o) {
    switch (S) {
        case 1: det_s<1>(T, a, h, lam, Y, o); break;
        case 2: det_s<2>(T, a, h, lam, Y, o); break;
        case 3: det_s<3>(T, a, h, lam, Y, o); break;
        case 4: det_s<4>(T, a, h, lam, Y, o); break;
        case 5: det_s<5>(T, a, h, lam, Y, o); break;
        default: det_s<6>(T, a, h, lam, Y, o);
    }
}
"""


@pytest.fixture(scope="module")
def lib():
    text = open(SRC).read()
    phi = re.search(r"DEV double phi_poly\(int r, double x\) \{.*?\n\}\n", text, re.S).group(0)
    i = text.index("DEV double qrcp(double x) {")
    part = text[i:text.index("/* ------------------------------------------------------------------ polynomial evaluators (FP64)", i)]
    os.makedirs(WORK, exist_ok=True)
    cpp, so = os.path.join(WORK, "fp64_math_host.cpp"), os.path.join(WORK, "fp64_math_host.so")
    with open(cpp, "w") as f:
        f.write(SHIM + phi + part + TAIL)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", cpp, "-o", so], check=True)
    return ctypes.CDLL(so)


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def test_reciprocal(lib):
    rng = np.random.Generator(np.random.PCG64(1))
    x = np.concatenate([np.exp(rng.uniform(-700, 700, 200000)) * rng.choice([-1.0, 1.0], 200000),
                        [1e-320, -1e-310, 2.0 ** -1022, 1.7e308, -1.7e308, np.inf, -np.inf, 1.0, 2.0, 1e-300, 1e300]])
    y = np.empty_like(x)
    lib.h_qrcp(ptr(x), ptr(y), ctypes.c_long(len(x)))
    with np.errstate(over="ignore", divide="ignore"):
        want = 1.0 / x
    fine = np.isfinite(want) & (np.abs(want) > 1e-300)
    assert (np.abs(y[fine] - want[fine]) <= 2.3e-16 * np.abs(want[fine])).all()  # one ulp
    assert np.array_equal(y[~fine], want[~fine])


@pytest.mark.parametrize("r", [0, 1, 2, 3])
def test_transform_and_weight(lib, r):
    from math import comb, factorial
    x = np.concatenate([np.linspace(1e-9, 1.0 - 1e-9, 4001), [0.5, np.nextafter(0.5, 0), 2.0 ** -40]])
    t, tm, w = (np.empty_like(x) for _ in range(3))
    lib.h_transform(r, ptr(x), ptr(t), ptr(tm), ptr(w), ctypes.c_long(len(x)))
    c = factorial(2 * r + 1) / factorial(r) ** 2
    phi = c * sum(comb(r, i) * (-1) ** i * x ** (r + i + 1) / (r + i + 1) for i in range(r + 1)) if r else x
    assert np.abs(t - phi).max() < 2e-13 and np.abs(t + tm - 1).max() < 3e-16  # the plain sum loses three digits near 1
    assert (np.abs(w - c * (x * (1 - x)) ** r) <= 1e-14 * c).all()


@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 6])
def test_determinant_with_and_without_zeroed_coordinates(lib, S):
    rng = np.random.Generator(np.random.PCG64(S))
    for Y in {0, 1, (1 << S) - 1, 2 % (1 << S), (1 << (S - 1)) | 1}:
        for lam in (0.0, 0.25, 0.7):
            t = rng.uniform(0, 1, S)
            t[[j for j in range(S) if (Y >> j) & 1]] = 0.0
            Tj = t * (1 - t)
            H = rng.uniform(-3, 3, (S, S))
            H = H + H.T
            g = rng.uniform(-3, 3, S)
            A = np.diag((1 - 2 * t) * g) + Tj[:, None] * H
            h = np.array([H[j, k] for j in range(S) for k in range(j, S)])
            o = np.zeros(2)
            a = np.ascontiguousarray(np.diag(A))
            lib.h_det(S, ptr(Tj), ptr(a), ptr(h), ctypes.c_double(lam), ctypes.c_uint(Y), ptr(o))
            want = np.linalg.det(np.eye(S) - 1j * lam * A)
            scale = np.prod(1 + lam * np.abs(A).sum(axis=1))  # Hadamard-like size of the terms
            assert abs(complex(*o) - want) <= 1e-14 * S * scale, (S, Y, lam)


def test_default_points_per_thread():
    """Passes that leave the launch shape open take the scratch of the shape they stand for: equal chunks, half the points
    below 6 items per SM (152), a quarter below one after that, an even number in mixed precision."""
    cfg = W.CONFIG3
    prep = api.prepare(T.compile_integral(cfg.topology, T.zero_invariants_of(cfg.topology, cfg.point)), cfg.kin,
                       cfg.order_min, cfg.order_max)
    ns = prep.info.n_sectors

    def scratch(n, m, prec, P=0):
        return api.scratch_bytes(prep, api.make_pass(n, [pow(76, j, n) or 1 for j in range(6)], m, 3, prec, points_per_thread=P))

    for prec, n, m, points in ((N.QMC_PREC_MIXED, 3001, 16, 12), (N.QMC_PREC_MIXED, 1021, 16, 4), (N.QMC_PREC_MIXED, 1048573, 16, 16),
                               (N.QMC_PREC_MIXED, 37, 1, 2), (N.QMC_PREC_FP64, 1021, 16, 4), (N.QMC_PREC_FP64, 4093, 16, 8),
                               (N.QMC_PREC_FP64, 1100, 1, 2), (N.QMC_PREC_FP64, 257, 1, 1)):
        items = ns * m * -(-n // (128 * points))
        assert scratch(n, m, prec) == scratch(n, m, prec, points) and items > 0, (prec, n, m)
