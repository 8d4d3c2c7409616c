"""The FP64 integrand's value and the eps-coefficient of its logarithm at one deformed point (`eval_G` in csrc/qmc_dev.cuh),
cut out as written and compiled for the host, over the whole range of its factors: the moduli of U and of q_j = 1 - i d_j
share a logarithm and a reciprocal where their product is moderate and must not overflow where it is not (d_j is
proportional to the scale of the kinematics, which is the user's choice of units, and |B_j| goes up to 64).

Reference: every factor by itself in logarithms with numpy.  Tolerance: the logarithms carry 4e-16 each, times the sum of
their sizes; G0 is compared through its logarithm."""
import ctypes
import os
import re
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from test_device_math_host import SHIM as SHIM_LOG

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WORK = os.path.join(ROOT, "tests", "_gen_build")
CSRC = os.path.join(ROOT, "paper_1508_02512_gb300", "csrc")

SHIM = r"""
#include <cstdlib>
#include "qmc_internal.h"
using std::abs;
#define __device__
#define __noinline__ static
struct cd { double x, y; };
DEV cd mk(double x, double y) { return cd{x, y}; }
DEV cd csub(cd a, cd b) { return cd{a.x - b.x, a.y - b.y}; }
DEV cd cscale(cd a, double s) { return cd{a.x * s, a.y * s}; }
DEV cd cmul(cd a, cd b) { return cd{fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x)}; }
static inline int __double2hiint(double d) { return (int)(__double_as_longlong(d) >> 32); }
DEV double rcp_seed(double x) { return (1.0 + (x > 0 ? 1 : -1) * 9.5367431640625e-7) / x; }
"""

TAIL = r"""
template <int S> struct Given { /* an evaluator that returns what it is given */
    const double *gv, *hv;
    cd u, f;
    void UFr(unsigned, const double *, double &, double &) const {}
    void GH(unsigned, const double *, double *g, double *h) const {
        for (int j = 0; j < S; ++j) g[j] = gv[j];
        for (int p = 0; p < S * (S + 1) / 2; ++p) h[p] = hv[p];
    }
    void UFc(unsigned, const cd *, bool, cd &U, cd &F) const { U = u; F = f; }
};
template <int S>
static void run(const int *A, const int *B, const int *e, const double *tt, const double *ttm, const double *Lt, double lam,
                const double *g, const double *h, const double *uf, double *out) {
    PackedSector s;
    std::memset(&s, 0, sizeof(s));
    s.D = 0.75;
    for (int j = 0; j < S; ++j) {
        s.A[j] = A[j];
        s.B[j] = B[j];
        s.sigma += A[j] == -1;
        qmc_sec.B[j] = B[j];
        qmc_sec.rB[j] = 1.0 / B[j];
    }
    const Given<S> P{g, h, mk(uf[0], uf[1]), mk(uf[2], uf[3])};
    cd G0, X;
    uint32_t fails = 0;
    eval_G<S>(s, P, 0u, tt, ttm, Lt, lam, true, Exps{e[0], e[1], e[2], e[3]}, G0, X, fails);
    out[0] = G0.x;
    out[1] = G0.y;
    out[2] = X.x;
    out[3] = X.y;
}
extern "C" void h_init() { logtab_init(); }
extern "C" void h_eval(int S, const int *A, const int *B, const int *e, const double *tt, const double *ttm, const double *Lt,
                       double lam, const double *g, const double *h, const double *uf, double *out) {
    if (S == 2) run<2>(A, B, e, tt, ttm, Lt, lam, g, h, uf, out);
    else if (S == 3) run<3>(A, B, e, tt, ttm, Lt, lam, g, h, uf, out);
    else run<6>(A, B, e, tt, ttm, Lt, lam, g, h, uf, out);
}
"""


def cut(text, start, end):
    i = text.index(start)
    return text[i:text.index(end, i)]


@pytest.fixture(scope="module")
def lib():
    text = open(os.path.join(CSRC, "qmc_dev.cuh")).read()
    logs = re.search(r"/\* -+ table-driven FP64 log and atan2 \*/(.*?)/\* principal log \*/", text, re.S).group(1)
    parts = [SHIM_LOG, SHIM, logs, cut(text, "DEV double arg_mi0(cd z)", "\n"), "\n",
             cut(text, "DEV double phi_poly(int r, double x) {", "\n}\n") + "\n}\n",
             cut(text, "DEV double qrcp(double x) {",
                 "/* ------------------------------------------------------------------ polynomial evaluators (FP64)"),
             "DEV double ipow(double, int) { return 0; }\n",
             cut(text, "/* ------------------------------------------------------------------ sector integrand */",
                 "/* w(x) * (sector integrand) at x, as series slots"), TAIL]
    os.makedirs(WORK, exist_ok=True)
    cpp, so = os.path.join(WORK, "fp64_range_host.cpp"), os.path.join(WORK, "fp64_range_host.so")
    with open(cpp, "w") as f:
        f.write("".join(parts))
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-I", CSRC, cpp, "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.h_init()
    return L


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def clog(z):
    """log z from the FP64 square of its modulus, as the integrand takes it (x x + y y, both roundings done exactly): below
    1e-154 that square is subnormal and holds fewer digits, in the kernel as here"""
    y2 = Fraction(float(Fraction(z.imag) ** 2))
    return 0.5 * np.log(float(Fraction(z.real) ** 2 + y2)) + 1j * np.arctan2(z.imag, z.real)


# size of the gradient; |U|; the largest |B_j|: the ordinary case, units of 1e4 to 1e60, large exponents, both
@pytest.mark.parametrize("size,usize,bmax", [(1.0, 1.0, 2), (1e4, 1e8, 2), (1e11, 1e22, 2), (1e20, 1e-40, 1), (1e60, 1e80, 2),
                                             (30.0, 1.0, 64), (300.0, 1e3, 64), (1e8, 1e-9, 64), (1e60, 1.0, 64),
                                             (1e-30, 1e-150, 64), (1.0, 1e-161, 3)])
@pytest.mark.parametrize("S", [2, 3, 6])
def test_value_and_logarithm(lib, S, size, usize, bmax):
    rng = np.random.Generator(np.random.PCG64(S * 1000 + bmax))
    for trial in range(40):
        t = rng.uniform(0.05, 0.95, S)
        g = size * rng.uniform(0.3, 3, S) * rng.choice([-1, 1], S)
        hess = np.diag(size * rng.uniform(0.0, 0.2, S) * np.sign((1 - 2 * t) * g))  # adds to the diagonal: no cancellation
        A = rng.choice([-1, -1, 0, 0, 1, 2], S).astype(np.int32)
        B = rng.integers(-bmax, bmax + 1, S).astype(np.int32)
        B[(A == -1) & (B == 0)] = -1
        if trial == 0:
            A[:], B[:] = -1, bmax
        if trial == 1:
            A[:], B[:] = -1, -bmax
        e = np.array([int(rng.integers(-2, 3)), int(rng.integers(2, 9)), int(rng.integers(1, 4)), int(rng.integers(1, 5))], np.int32)
        if usize > 1e50 or usize < 1e-50:
            e[0] = 0  # keeps G0 itself in range
        U = usize * complex(rng.uniform(0.3, 2), rng.uniform(-1, 1))
        F = size * complex(rng.uniform(-1, 1), -rng.uniform(0.1, 1))
        lam, Lt = 0.5, np.log(t)
        h = np.array([hess[j, k] for j in range(S) for k in range(j, S)])
        out = np.zeros(4)
        tm = 1 - t
        uf = np.array([U.real, U.imag, F.real, F.imag])
        lib.h_eval(S, ptr(A), ptr(B), ptr(e), ptr(t), ptr(tm), ptr(Lt), ctypes.c_double(lam), ptr(g), ptr(h), ptr(uf), ptr(out))
        q = 1 - 1j * (lam * tm * g)
        pivots = 1 - 1j * lam * ((1 - 2 * t) * g + t * tm * np.diag(hess))
        parts = [e[1] * clog(U), -e[3] * clog(F)] + [B[j] * clog(q[j]) for j in range(S)]
        parts += [B[j] * Lt[j] for j in range(S) if A[j] != -1]
        want = sum(parts)
        scale = sum(abs(p) for p in parts) + 1
        assert abs(out[2] - want.real) <= 4e-15 * scale and abs(out[3] - want.imag) <= 4e-15 * scale, (trial, out, want)
        lg = [clog(p) for p in pivots] + [e[0] * clog(U), -e[2] * clog(F), np.log(0.75)]
        lg += [A[j] * clog(q[j]) for j in range(S)] + [A[j] * Lt[j] for j in range(S) if A[j] > 0]
        lw = sum(lg)
        up = sum(max(p.real, 0.0) for p in map(complex, lg))
        down = sum(min(p.real, 0.0) for p in map(complex, lg))
        if up > 600 or down < -600:
            continue  # a partial product of G0 itself may leave the range, in whatever order it is taken
        r = complex(out[0], out[1]) / np.exp(lw)
        assert abs(r - 1) <= 1e-15 * (sum(abs(p) for p in lg) + 40), (trial, r)


@pytest.mark.gpu
def test_integration_in_large_units():
    """The non-planar double box with every invariant times 1e20: at the first lambda d_j is of that size, the sign check
    fails, and lambda is halved until the contour fits; the result is kappa^-(eF0 + eF1 eps) times the plain one."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import math

    import workloads as W
    from paper_1508_02512_gb300 import _native as N
    from paper_1508_02512_gb300 import api
    from paper_1508_02512_gb300 import tables as T
    cfg, kappa = W.CONFIG3, 1e20
    meta, _ = T.read_table(T.compile_integral(cfg.topology, T.zero_invariants_of(cfg.topology, cfg.point)))
    got = []
    for scale in (1.0, kappa):
        c = api.Context()
        i = c.load_sectors(T.compile_integral(cfg.topology, T.zero_invariants_of(cfg.topology, cfg.point)))
        c.set_kinematics(i, scale * np.asarray(cfg.kin), cfg.order_min, cfg.order_max)
        r = c.integrate(i, rel_tol=1e-2, precision=N.QMC_PREC_FP64, max_halvings=100)
        c.close()
        assert r.status == N.QMC_OK and r.nonfinite_sectors == 0
        got.append(api.result_arrays(r))
    (v, e), (vk, ek) = got
    eF0, eF1 = meta["eF"]
    lk = -eF1 * math.log(kappa)
    for k in range(len(v)):
        f = [kappa ** -eF0 * lk ** j / math.factorial(j) for j in range(k + 1)]
        want = sum(f[j] * v[k - j] for j in range(k + 1))
        tol = 5 * (np.hypot(*ek[k]) + sum(abs(f[j]) * np.hypot(*e[k - j]) for j in range(k + 1)))
        assert abs(vk[k] - want) <= tol, (k, vk[k], want, tol)
