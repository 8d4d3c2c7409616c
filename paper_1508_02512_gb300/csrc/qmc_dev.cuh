#pragma once
/*
 * GB300 (sm_103a) kernels of the quasi-Monte Carlo sector integrator.
 *
 * Li, Wang, Yan, Zhao, "Efficient Numerical Evaluation of Feynman Integrals", Chin. Phys. C 40 (2016) 033103.
 *
 * qmc_eval_kernel (persistent, one launch per sector class): blocks take work items from an atomic counter;
 *   an item is (sector, shift, chunk of blockDim * P consecutive lattice indices).  The block stages the
 *   sector's polynomial terms into shared memory (one copy per sector change), each thread walks P lattice
 *   points i = i0 + p * blockDim with integer index arithmetic (Eq. 17: x = {i z / n + Delta}), evaluates
 *   the sector integrand series (periodising transform Eq. 21, contour deformation Eq. 14 with its Jacobian,
 *   endpoint subtraction Eqs. 10-12, eps expansion) and accumulates it with Kahan compensation; the block
 *   reduces with warp shuffles and writes one partial per item and slot.
 * qmc_finalize_kernel: one warp per (sector, shift) sums that pair's item partials in a fixed order
 *   (compensated), so results do not depend on which block ran which item (Eqs. 16 and 18).
 * qmc_points_kernel: the same per-point device code on explicit lattice indices (sampled checks).
 *
 * The FP64 path is bound by the FP64 pipe, the FP32 path by instruction issue and the FP32 pipe's operand ports (no dense
 * contraction, nothing streamed from HBM), so no tensor cores or TMA are used: tables live in shared memory, points are generated, outputs are a few KB.
 *
 * This header holds device code only, so that it also compiles at run time (NVRTC) together with the
 * polynomial code generated for one family of sector tables; the host launchers are in qmc_device.cuh.
 */
#ifndef __CUDACC_RTC__
#include <math.h>
#include <stdint.h>
#endif

#include "qmc_internal.h"

#define DEV __device__ __forceinline__
#define QMC_PI 3.141592653589793

/* ------------------------------------------------------------------ complex double */
struct cd {
    double x, y;
};
DEV cd mk(double x, double y) { return cd{x, y}; }
DEV cd csub(cd a, cd b) { return cd{a.x - b.x, a.y - b.y}; }
DEV cd cscale(cd a, double s) { return cd{a.x * s, a.y * s}; }
DEV cd cmul(cd a, cd b) { return cd{fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x)}; }
DEV double ipow(double v, int e) {
    if (e == 0) return 1.0;
    double r = v;
    for (int i = e < 0 ? -e : e; i > 1; --i) r *= v;
    return e < 0 ? __drcp_rn(r) : r;
}
/* ------------------------------------------------------------------ table-driven FP64 log and atan2 */
/* Logarithm after Tang (P. T. P. Tang, ACM Trans. Math. Softw. 16 (1990) 378): x = 2^e m with m in [1, 2);
   c = 1 + k/128 is the grid point nearest m (k = 0..128); log x = e ln2 + log c + log1p(r) with r = (m - c)/c,
   |r| <= 2^-8, and log1p(r) from its Taylor series through r^7 (the first omitted term is below 2^-67).  m - c
   is exact.  For k >= 64 the split is recentred on 1, log x = (e + 1) ln2 + log(c/2) + log1p(r), so that
   arguments just below 1 meet no cancellation between e ln2 and log c.
   Arctangent by the same table-driven reduction: for 0 <= u = lo/hi <= 1 and the grid point c = k/128 nearest u,
   atan u = atan c + atan(d) with d = (u - c)/(1 + u c) = (lo - c hi)/(hi + c lo), |d| <= 2^-8 + 2^-20, and atan d
   from its Taylor series through d^7 (omitted term below 2^-77); k comes from an FP32 estimate of u, which only
   has to land on the nearest or a neighbouring grid point.  Octants follow from the signs and the swap.
   The tables {1/c, log c} and {k/128, atan(k/128)} are filled once per block (library functions) by
   logtab_init and read from shared memory; arguments outside the fast paths go to the library. */
struct LogTable {
    double inv_c[129];
    double log_c[129];
    double grid[129];
    double atan_c[129];
};
static __shared__ LogTable qmc_logtab;

/* every thread of the block calls it; a __syncthreads() must follow before the first qlog / qatan2 */
DEV void logtab_init() {
    for (int k = threadIdx.x; k <= 128; k += blockDim.x) {
        const double c = 1.0 + k / 128.0;
        qmc_logtab.inv_c[k] = 1.0 / c;
        qmc_logtab.log_c[k] = k < 64 ? log(c) : log(0.5 * c);
        qmc_logtab.grid[k] = k / 128.0;
        qmc_logtab.atan_c[k] = atan(k / 128.0);
    }
}

DEV double qatan2(double y, double x) {
    /* magnitudes compare as the integers of their bit patterns (FP64 compares would run on the FP64 pipe) */
    const double a = fabs(x), b = fabs(y);
    const long long ba = __double_as_longlong(a), bb = __double_as_longlong(b);
    const bool swap = bb > ba;
    const double hi = swap ? b : a, lo = swap ? a : b;
    const long long bh = swap ? bb : ba;
    if (!(bh > __double_as_longlong(1e-30) && bh < __double_as_longlong(1e30)))
        return atan2(y, x); /* zero, tiny, huge or not a number */
    const int k = min(max(__float2int_rn(128.f * __fdividef((float)lo, (float)hi)), 0), 128);
    const double c = qmc_logtab.grid[k];
    const double d = fma(-c, hi, lo) * __drcp_rn(fma(c, lo, hi));
    const double d2 = d * d;
    double q = fma(d2, -1.0 / 7.0, 1.0 / 5.0);
    q = fma(q, d2, -1.0 / 3.0);
    const double th = qmc_logtab.atan_c[k] + fma(d * d2, q, d);
    /* the octant: th, pi/2 - th (swapped), pi - th (x < 0), pi/2 + th (both) */
    const bool neg = __double_as_longlong(x) < 0;
    const double base = swap ? 0.5 * QMC_PI : (neg ? QMC_PI : 0.0);
    return copysign(base + (swap != neg ? -th : th), y);
}

DEV double qlog(double x) {
    const long long b = __double_as_longlong(x);
    const long long be = b >> 52; /* biased exponent of a positive number; <= 0 for x <= 0 */
    if (be <= 0 || be >= 2047) return log(x);
    const int k = (int)((((b >> 44) & 0xFF) + 1) >> 1);
    const double m = __longlong_as_double((b & 0x000FFFFFFFFFFFFFLL) | 0x3FF0000000000000LL);
    const double c = __longlong_as_double(0x3FF0000000000000LL + ((long long)k << 45));
    const double r = (m - c) * qmc_logtab.inv_c[k];
    double q = fma(r, 1.0 / 7.0, -1.0 / 6.0);
    q = fma(q, r, 1.0 / 5.0);
    q = fma(q, r, -1.0 / 4.0);
    q = fma(q, r, 1.0 / 3.0);
    q = fma(q, r, -0.5);
    const double p = fma(r * r, q, r);
    const double e = (double)(int)(be - 1023 + (k >= 64));
    const double LN2 = 0.6931471805599453, LN2_LO = 2.3190468138462996e-17; /* ln 2 = LN2 + LN2_LO */
    return fma(e, LN2, qmc_logtab.log_c[k]) + fma(e, LN2_LO, p);
}

/* principal log */
/* its imaginary part is qatan2 for U and the q_j; for F - i0 a negative real F lies at -pi */
DEV double arg_mi0(cd z) { return z.y == 0.0 ? (z.x < 0.0 ? -QMC_PI : 0.0) : qatan2(z.y, z.x); }

/* ------------------------------------------------------------------ periodising transform (Eq. 21, order r) */
/* t = phi_r(x), tm = phi_r(1-x) = 1 - t, w = phi_r'(x); phi_r' = c_r x^r (1-x)^r, c_r = (2r+1)!/(r!)^2 */
DEV double phi_poly(int r, double x) {
    switch (r) {
        case 0: return x;
        case 1: return x * x * fma(-2.0, x, 3.0);
        case 2: return x * x * x * fma(x, fma(6.0, x, -15.0), 10.0);
        default: {
            const double x2 = x * x;
            return x2 * x2 * fma(x, fma(x, fma(-20.0, x, 70.0), -84.0), 35.0);
        }
    }
}
/* phi is evaluated on the smaller of x and 1-x only; phi_r(1-x) = 1 - phi_r(x) gives the other side, which is
   >= 1/2 and therefore exact to rounding */
DEV void transform(int r, double x, double &t, double &tm, double &w) {
    const double y = 1.0 - x;
    const bool lo = x <= 0.5;
    const double p = phi_poly(r, lo ? x : y);
    const double q = 1.0 - p;
    t = lo ? p : q;
    tm = lo ? q : p;
    const double xy = x * y;
    switch (r) {
        case 0: w = 1.0; break;
        case 1: w = 6.0 * xy; break;
        case 2: w = 30.0 * xy * xy; break;
        default: w = 140.0 * xy * xy * xy; break;
    }
}

/* ------------------------------------------------------------------ polynomials from shared memory */
DEV uint64_t term_exps(const PackedTerm &T) { return *reinterpret_cast<const uint64_t *>(T.e); }

/* sum_a c_a prod_j t_j^{e_aj}: the monomial starts from its first factor and the coefficient enters through
   one FMA into the accumulator; exponents are warp-uniform (every lane reads the same term) */
template <int S>
DEV double poly_r(const PackedTerm *__restrict__ T, int n, const double *t) {
    double acc = 0.0;
    for (int a = 0; a < n; ++a) {
        const double c = T[a].c;
        const uint64_t ew = term_exps(T[a]);
        if (ew == 0) {
            acc += c;
            continue;
        }
        double m = 1.0;
        bool have = false;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            int e = (int)((ew >> (8 * j)) & 0xffu);
            if (e > 0) {
                if (!have) {
                    m = t[j];
                    have = true;
                    --e;
                }
                for (int k = 0; k < e; ++k) m *= t[j];
            }
        }
        acc = fma(c, m, acc);
    }
    return acc;
}

template <int S>
DEV cd poly_c(const PackedTerm *__restrict__ T, int n, const cd *z) {
    cd acc = mk(0.0, 0.0);
    for (int a = 0; a < n; ++a) {
        const double c = T[a].c;
        const uint64_t ew = term_exps(T[a]);
        if (ew == 0) {
            acc.x += c;
            continue;
        }
        cd m = mk(1.0, 0.0);
        bool have = false;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            int e = (int)((ew >> (8 * j)) & 0xffu);
            if (e > 0) {
                if (!have) {
                    m = z[j];
                    have = true;
                    --e;
                }
                for (int k = 0; k < e; ++k) m = cmul(m, z[j]);
            }
        }
        acc.x = fma(c, m.x, acc.x);
        acc.y = fma(c, m.y, acc.y);
    }
    return acc;
}

/* ------------------------------------------------------------------ reciprocals, powers and x on the FP64 pipe
   The FP64 kernels are bound by the FP64 pipe alone (2 lanes per clock and SM: one warp instruction takes 16 cycles
   of it, in which the SM can issue 64 others).  It also executes FP64 compares and integer conversions, so the code
   below compares bit patterns, keeps small integers as doubles, and counts operations rather than instructions. */
DEV double rcp_seed(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}
/* 1/x from an approximation r good to some 20 bits, by one step of Householder's third-order iteration: with
   e = 1 - x r, 1/x = r (1 + e + e^2 + ...) and the first term left out is e^3 < 2^-57, so
   the result is within 0.51 units in the last place (0.508 found over 2e6 arguments).  Three FMAs; the correctly
   rounded __drcp_rn takes as much of the FP64 pipe as 5.3 of them (measured), and is left for arguments whose
   reciprocal could leave the normal range. */
DEV double qrcp(double x) {
    const unsigned be = ((unsigned)__double2hiint(x) >> 20) & 0x7FFu; /* biased exponent */
    if (be - 24u > 1998u) return __drcp_rn(x);
    const double r = rcp_seed(x);
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
/* v^e for e >= 1, inv^|e| for e < 0, inv = 1/v */
DEV cd cpow_inv(cd v, cd inv, int e) {
    const cd b = e < 0 ? inv : v;
    cd r = b;
    for (int i = e < 0 ? -e : e; i > 1; --i) r = cmul(r, b);
    return r;
}
/* a > 0 (false for NaN), by the bit pattern */
DEV bool is_positive(double a) {
    const long long b = __double_as_longlong(a);
    return b > 0 && b <= 0x7FF0000000000000LL;
}
/* transform for the FP64 kernels: t, tm = 1 - t, and xy = x (1 - x), whose product over the variables gives the
   weight prod_j phi_r'(x_j) = c_r^S (prod_j xy_j)^r at once (weight64) */
DEV void transform64(int r, double x, double &t, double &tm, double &xy) {
    const double y = 1.0 - x;
    const bool lo = __double2hiint(x) < 0x3FE00000; /* 0 < x < 1/2 */
    const double p = phi_poly(r, lo ? x : y);
    const double q = 1.0 - p;
    t = lo ? p : q;
    tm = lo ? q : p;
    xy = x * y;
}
template <int S>
DEV double weight64(int r, double xy) {
    double c = 1.0; /* c_r^S, folded at compile time for each r */
    switch (r) {
        case 0: return 1.0;
        case 1:
#pragma unroll
            for (int j = 0; j < S; ++j) c *= 6.0;
            return c * xy;
        case 2:
#pragma unroll
            for (int j = 0; j < S; ++j) c *= 30.0;
            return c * (xy * xy);
        default:
#pragma unroll
            for (int j = 0; j < S; ++j) c *= 140.0;
            return c * (xy * xy * xy);
    }
}

/* The exponents' eps parts B_j of the staged sector and their reciprocals as doubles (stage_sector fills them):
   conversions and divisions run on the FP64 pipe, so they are made once per block and sector. */
struct SectorConst {
    double B[8], rB[8];
};
static __shared__ SectorConst qmc_sec;

/* ------------------------------------------------------------------ det(I - i lam A), A = D + T H
   A_jk = delta_jk (1 - 2 t_j) g_j + T_j h_jk with T_j = t_j (1 - t_j) and h the symmetric Hessian of F (packed upper
   triangle): a[j] = A_jj, and the off-diagonal entries are those of a symmetric matrix with row j scaled by T_j.
   T^{-1/2} A T^{1/2} is symmetric, so I - i lam A is similar to a complex symmetric matrix whose Hermitian part is the
   identity: every Schur complement keeps a Hermitian part >= 1 and elimination needs no pivoting.  Carried out
   without the square roots, on s_j = M_jj and Z_jk with M_jk = T_j Z_jk:
     s_i -= T_i (T_k / s_k) Z_ki^2,   Z_ij -= (T_k / s_k) Z_ki Z_kj,   i, j > k.
   T_k = 0 (a coordinate of the zeroed subset Y) leaves nothing to eliminate.  The first step's Z are imaginary, so its
   products are real.  About 290 FP64 operations for S = 6 (fewer with zeroed coordinates) instead of the 600 of a
   pivoted elimination on the full matrix: with the shorter series and logarithms of point_integrand, the FP64 pass of
   the non-planar double box (n = 16381, 16 shifts) went from 54.7 to 34.3 ms, the massive box's (n = 262139) from 5.69
   to 4.92 ms. */
template <int S>
DEV cd det_deform(const double (&T)[S], const double (&a)[S], const double *h, double lam, unsigned Y) {
    auto at = [](int i, int j) { return i * S - i * (i - 1) / 2 + (j - i); }; /* i <= j */
    if constexpr (S == 1) {
        return mk(1.0, -lam * a[0]);
    } else if constexpr (S == 2) {
        const double e2 = fma(a[0], a[1], -(T[0] * T[1]) * (h[1] * h[1]));
        return mk(fma(-lam * lam, e2, 1.0), -lam * (a[0] + a[1]));
    } else if constexpr (S == 3) {
        /* det(I + cA) = 1 + c tr A + c^2 E2(A) + c^3 det A with c = -i lam */
        const double h01 = h[at(0, 1)], h02 = h[at(0, 2)], h12 = h[at(1, 2)];
        const double t01 = T[0] * T[1], p01 = t01 * (h01 * h01), p02 = T[0] * T[2] * (h02 * h02);
        const double p12 = T[1] * T[2] * (h12 * h12);
        const double m01 = fma(a[0], a[1], -p01);
        const double e2 = fma(a[0], a[2], -p02) + fma(a[1], a[2], -p12) + m01;
        const double x3 = t01 * T[2] * (h01 * h02 * h12);
        const double dt = fma(m01, a[2], fma(-a[0], p12, fma(-a[1], p02, x3 + x3)));
        const double l2 = lam * lam;
        return mk(fma(-l2, e2, 1.0), lam * fma(l2, dt, -(a[0] + a[1] + a[2])));
    } else {
        cd s[S], Z[S * (S + 1) / 2];
#pragma unroll
        for (int j = 0; j < S; ++j) s[j] = mk(1.0, -lam * a[j]);
#pragma unroll
        for (int i = 1; i < S; ++i)
#pragma unroll
            for (int j = i + 1; j < S; ++j) Z[at(i, j)] = mk(0.0, -lam * h[at(i, j)]);
        cd det = s[0];
        if (!(Y & 1u)) {
            /* Z_0i Z_0j = -lam^2 h_0i h_0j; rho = lam^2 T_0 / s_0 with Re s_0 = 1 */
            const double f = (lam * lam) * T[0] * qrcp(fma(s[0].y, s[0].y, 1.0));
            const cd rho = mk(f, -s[0].y * f);
#pragma unroll
            for (int i = 1; i < S; ++i) {
                const double q = T[i] * (h[at(0, i)] * h[at(0, i)]);
                s[i].x = fma(rho.x, q, s[i].x);
                s[i].y = fma(rho.y, q, s[i].y);
#pragma unroll
                for (int j = i + 1; j < S; ++j) {
                    const double hh = h[at(0, i)] * h[at(0, j)];
                    Z[at(i, j)].x = rho.x * hh;
                    Z[at(i, j)].y = fma(rho.y, hh, Z[at(i, j)].y);
                }
            }
        }
#pragma unroll
        for (int k = 1; k < S; ++k) {
            det = cmul(det, s[k]);
            if (k + 1 < S && !((Y >> k) & 1u)) {
                const double f = T[k] * qrcp(fma(s[k].x, s[k].x, s[k].y * s[k].y));
                const cd rho = mk(s[k].x * f, -s[k].y * f);
#pragma unroll
                for (int i = k + 1; i < S; ++i) {
                    const cd z = Z[at(k, i)], l = cmul(rho, z), m = cmul(l, z);
                    s[i].x = fma(-T[i], m.x, s[i].x);
                    s[i].y = fma(-T[i], m.y, s[i].y);
#pragma unroll
                    for (int j = i + 1; j < S; ++j) {
                        const cd w = Z[at(k, j)];
                        cd &v = Z[at(i, j)];
                        v.x = fma(-l.x, w.x, fma(l.y, w.y, v.x));
                        v.y = fma(-l.x, w.y, fma(-l.y, w.x, v.y));
                    }
                }
            }
        }
        return det;
    }
}

struct Exps {
    int eU0, eU1, eF0, eF1;
};

/* ------------------------------------------------------------------ polynomial evaluators (FP64)
   The integrand asks an evaluator for
     UFr(Y, t, U, F)          U~ and F~ at real t (undeformed sectors, Eqs. 7-8),
     GH(Y, t, g, h)           g_j = dF~/dt_j and h_p = d2F~/dt_j dt_k (p over j <= k, row-major upper triangle) at
                              real t, the inputs of the deformation of Eq. 14,
     UFc(Y, z, needU, U, F)   U~ (1 when needU is false) and F~ at the deformed point z,
   where the coordinates in the subset Y (bit j = variable j) of the endpoint subtraction (Eqs. 10-12) are zero, and
     exps(J)               the powers eU0 + eU1 eps and eF0 + eF1 eps of U~ and 1/F~.
   TabPol walks the staged term table (and ignores Y: zero coordinates make those terms vanish); the generated
   FP64 evaluator (run-time compiled per family) holds each sector's monomials, per zeroed subset without the
   terms that vanish there, as straight-line code and reads only the coefficients from the same table. */
template <int S>
struct TabPol {
    const PackedTerm *T;
    const PackedSector *s;
    DEV static TabPol make(const PackedTerm *T, const PackedSector &s, int) { return TabPol{T, &s}; }
    DEV static Exps exps(const Job &J) { return Exps{J.eU0, J.eU1, J.eF0, J.eF1}; }
    DEV void UFr(unsigned, const double *t, double &U, double &F) const {
        U = poly_r<S>(T, s->nU, t);
        F = poly_r<S>(T + s->nU, s->nF, t);
    }
    DEV void GH(unsigned, const double *t, double *g, double *h) const {
        const PackedTerm *TG = T + s->nU + s->nF;
        const PackedTerm *TH = TG + s->nG;
#pragma unroll
        for (int j = 0; j < S; ++j) g[j] = poly_r<S>(TG + s->gstart[j], s->gstart[j + 1] - s->gstart[j], t);
#pragma unroll
        for (int p = 0; p < S * (S + 1) / 2; ++p) h[p] = poly_r<S>(TH + s->hstart[p], s->hstart[p + 1] - s->hstart[p], t);
    }
    DEV void UFc(unsigned, const cd *z, bool needU, cd &U, cd &F) const {
        U = needU ? poly_c<S>(T, s->nU, z) : mk(1.0, 0.0);
        F = poly_c<S>(T + s->nU, s->nF, z);
    }
};

/* ------------------------------------------------------------------ sector integrand */
template <bool B, class T, class F>
struct Select {
    typedef F type;
};
template <class T, class F>
struct Select<true, T, F> {
    typedef T type;
};
template <bool B>
struct EnableIf {};
template <>
struct EnableIf<true> {
    typedef void type;
};


/* Products over the q_j = 1 - i d_j of a deformed point, where they could leave the range of a double.  d_j carries the
   scale of the kinematics (F~ is not normalised): before lambda has been halved far enough it can be anything.  The usual
   case is inlined in eval_G; these are functions of their own, because the compiler would execute both sides of a short
   branch, and the FP64 pipe is the bound (non-planar double box, n = 1021, one shift: 303 us without them, 318-323 with
   both forms inlined, 304 as they are). */
DEV int exponent(double x) { return (int)(((unsigned)__double2hiint(x) >> 20) & 0x7FFu) - 1023; } /* 1024: infinity, NaN */
/* bound on log2(1 + d^2), on the integer pipes */
DEV int modulus_exponent(double d) {
    const int e = exponent(d);
    return e < 0 ? 1 : 2 * e + 3;
}
template <int S>
struct Contour {
    double d[S];
};
/* G prod_j q_j^{A_j}, factor by factor */
template <int S>
__device__ __noinline__ cd times_q(const PackedSector &s, Contour<S> c, cd G) {
#pragma unroll
    for (int j = 0; j < S; ++j) {
        for (int k = 0; k < s.A[j]; ++k) G = cmul(G, mk(1.0, -c.d[j]));
        for (int k = 0; k > s.A[j]; --k) {
            const double f = __drcp_rn(fma(c.d[j], c.d[j], 1.0));
            G = cmul(G, mk(f, c.d[j] * f));
        }
    }
    return G;
}
/* v^k to the product num / dnm: its mantissa in [1, 2), and its exponent to e2 (zero, infinity and NaN as they are) */
DEV void mul_mantissa(double &num, double &dnm, int &e2, double v, int k) {
    if (exponent(v) == -1023) {
        v *= 18014398509481984.0; /* 2^54: subnormal numbers become normal */
        e2 -= 54 * k;
    }
    const int e = exponent(v);
    if (e > -1023 && e < 1024) {
        e2 += e * k;
        v = __longlong_as_double((__double_as_longlong(v) & 0x000FFFFFFFFFFFFFLL) | 0x3FF0000000000000LL);
    }
    for (int i = 0; i < k; ++i) num *= v;
    for (int i = 0; i > k; --i) dnm *= v;
}
/* eU1 log U2 + sum_j B_j log(1 + d_j^2) */
template <int S>
__device__ __noinline__ double log_moduli(const PackedSector &s, Contour<S> c, double U2, int eU1) {
    double num = 1.0, dnm = 1.0;
    int e2 = 0;
    mul_mantissa(num, dnm, e2, U2, eU1);
#pragma unroll
    for (int j = 0; j < S; ++j) mul_mantissa(num, dnm, e2, fma(c.d[j], c.d[j], 1.0), s.B[j]);
    return fma((double)e2, 0.6931471805599453, qlog(num * qrcp(dnm)));
}

/* G at the point tt (t with the subset Y zeroed): returns its eps^0 value G0 and, with needX, the eps-coefficient X of
   its logarithm, so that G(eps) = G0 exp(X eps) (Sec. II, Eq. 9 with the deformation of Eq. 14).  First the undeformed
   class, where everything is real. */
template <int S, class Pol>
DEV void eval_G(const PackedSector &s, const Pol &P, unsigned Y, const double *tt, const double *Lt, bool needX,
                const Exps &ex, double &G0, double &X) {
    double U, F;
    P.UFr(Y, tt, U, F);
    if (s.kind == 1) F = -F;
    double g = s.D * ipow(U, ex.eU0) * ipow(F, -ex.eF0);
#pragma unroll
    for (int j = 0; j < S; ++j)
        for (int k = 0; k < s.A[j]; ++k) g *= tt[j];
    G0 = g;
    X = 0.0;
    if (needX) {
        /* eU1 log U - eF1 log F as one logarithm: both are real and positive on this path */
        double x = qlog(ipow(U, ex.eU1) * ipow(F, -ex.eF1));
#pragma unroll
        for (int j = 0; j < S; ++j)
            if (s.A[j] != -1 && s.B[j] != 0) x = fma(qmc_sec.B[j], Lt[j], x);
        X = x;
    }
}

template <int S, class Pol>
DEV void eval_G(const PackedSector &s, const Pol &P, unsigned Y, const double *tt, const double *ttm, const double *Lt,
                double lam, bool needX, const Exps &ex, cd &G0, cd &X, uint32_t &fails) {
    double d[S];
    cd detJ;
    {
        double g[S], h[S * (S + 1) / 2];
        P.GH(Y, tt, g, h);
        double T[S], a[S];
        int p = 0;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            T[j] = tt[j] * ttm[j];
            a[j] = fma(ttm[j] - tt[j], g[j], T[j] * h[p]);
            d[j] = lam * ttm[j] * g[j];
            p += S - j;
        }
        detJ = det_deform<S>(T, a, h, lam, Y);
    }
    /* z_j = t_j q_j with q_j = 1 - i d_j */
    cd z[S];
#pragma unroll
    for (int j = 0; j < S; ++j) z[j] = mk(tt[j], -tt[j] * d[j]);
    cd U, F;
    P.UFc(Y, z, ex.eU0 != 0 || needX, U, F);
    fails += is_positive(F.y) ? 1u : 0u;
    const double F2 = fma(F.x, F.x, F.y * F.y);
    cd G = detJ;
    if (ex.eF0 != 0) {
        const double f = qrcp(F2);
        G = cmul(G, cpow_inv(F, mk(F.x * f, -F.y * f), -ex.eF0));
    }
    if (ex.eU0 > 0) {
        G = cmul(G, cpow_inv(U, U, ex.eU0));
    } else if (ex.eU0 < 0) {
        const double f = qrcp(fma(U.x, U.x, U.y * U.y));
        const cd iU = mk(U.x * f, -U.y * f);
        G = cmul(G, cpow_inv(iU, iU, -ex.eU0));
    }
    /* prod_j (t_j q_j)^{A_j}, t_j only for A_j >= 0: a product with q_j is two FMAs, and 1/q_j = (1 + i d_j)/(1 + d_j^2).
       The moduli 1 + d_j^2 share one reciprocal while their product stays below 2^200. */
    double re = s.D, den = 1.0;
    const cd G1 = G;
    int size = 0;
#pragma unroll
    for (int j = 0; j < S; ++j) {
        for (int k = 0; k < s.A[j]; ++k) {
            re *= tt[j];
            G = mk(fma(G.y, d[j], G.x), fma(-G.x, d[j], G.y));
        }
        for (int k = 0; k > s.A[j]; --k) {
            den *= fma(d[j], d[j], 1.0);
            G = mk(fma(-G.y, d[j], G.x), fma(G.x, d[j], G.y));
            size += modulus_exponent(d[j]);
        }
    }
    if (size > 200) {
        Contour<S> c;
#pragma unroll
        for (int j = 0; j < S; ++j) c.d[j] = d[j];
        G = times_q<S>(s, c, G1);
        den = 1.0;
    }
    if (s.sigma > 0) re *= qrcp(den);
    G0 = cscale(G, re);
    X = mk(0.0, 0.0);
    if (needX) {
        /* eU1 log U - eF1 log F + sum_j B_j log q_j (and B_j log t_j where A_j != -1).  The moduli of U and of the q_j
           share one logarithm while their product stays within 2^-1000 to 2^1000. */
        const double U2 = fma(U.x, U.x, U.y * U.y);
        double num = 1.0, dnm = 1.0, xr = 0.0;
        double xi = (double)ex.eU1 * qatan2(U.y, U.x);
        for (int k = 0; k < ex.eU1; ++k) num *= U2;
        for (int k = 0; k > ex.eU1; --k) dnm *= U2;
        size = abs(ex.eU1) * (abs(exponent(U2)) + 1);
#pragma unroll
        for (int j = 0; j < S; ++j) {
            if (s.B[j] != 0) {
                if (s.A[j] != -1) xr = fma(qmc_sec.B[j], Lt[j], xr);
                const double q2 = fma(d[j], d[j], 1.0);
                for (int k = 0; k < s.B[j]; ++k) num *= q2;
                for (int k = 0; k > s.B[j]; --k) dnm *= q2;
                size += abs(s.B[j]) * modulus_exponent(d[j]);
                xi = fma(-qmc_sec.B[j], qatan2(d[j], 1.0), xi);
            }
        }
        const double eF1 = (double)ex.eF1;
        double l;
        if (size > 1000) {
            Contour<S> c;
#pragma unroll
            for (int j = 0; j < S; ++j) c.d[j] = d[j];
            l = log_moduli<S>(s, c, U2, ex.eU1);
        } else {
            l = qlog(num * qrcp(dnm));
        }
        X.x = fma(0.5, fma(-eF1, qlog(F2), l), xr);
        X.y = fma(-eF1, arg_mi0(F), xi);
    }
}

/* w(x) * (sector integrand) at x, as series slots 0..M (slot n = coefficient of eps^(n - sigma)).
   Subtraction of Eq. (11) with alpha = -1 over the zeroed subsets Y of the singular set: with
   a_j(eps) = eps t_j^{-1 + B_j eps} = sum_{n >= 1} c_n eps^n, each singular variable turns G into a_j (G - G|_{t_j = 0}) +
   G|_{t_j = 0} / B_j.  The series a_j are made once per point.  Every variable outside Y brings a factor eps, so G_Y is
   needed to eps^(M - sigma + |Y|) only: its logarithm X is left out where that is zero, in particular at the point
   itself (Y empty) whenever the highest order wanted is eps^0. */
struct Subsets {
    int sigma, M;
    unsigned smask;
    /* highest order of eps to which G_Y is needed, count: the subset's bits in singular-variable numbering */
    DEV int need(unsigned count) const { return M - sigma + __popc(count); }
};

/* t, 1 - t, logarithms, weight and the series a_j of a point; false: the weight vanishes there */
template <int S, int MAXM>
DEV bool point_setup(const PackedSector &s, const double *x, int r, const Subsets &q, double (&t)[S], double (&tm)[S],
                     double (&Lt)[S], double (&a)[S][MAXM + 1], double &w) {
    bool bad = false;
#pragma unroll
    for (int j = 0; j < S; ++j) {
        double xy;
        transform64(r, x[j], t[j], tm[j], xy);
        w = j == 0 ? xy : w * xy;
        bad |= __double_as_longlong(x[j]) <= 0; /* the weight and t vanish only at x = 0: x < 1 after the wrap */
    }
    if (bad) return false;
    w = weight64<S>(r, w);
    int i = 0;
#pragma unroll
    for (int j = 0; j < S; ++j) {
        const bool sing = (q.smask >> j) & 1u;
        Lt[j] = 0.0;
        if (MAXM > 0 && q.M > 0 && (sing || s.B[j] != 0)) Lt[j] = qlog(t[j]);
        if (!sing) continue;
        a[i][0] = qmc_sec.rB[j]; /* the place of eps^0 holds 1/B_j */
        if (MAXM > 0 && q.M > 0) {
            double c = __drcp_rn(t[j]);
            const double bl = qmc_sec.B[j] * Lt[j];
#pragma unroll
            for (int n = 1; n <= MAXM; ++n) {
                if (n > q.M) break;
                a[i][n] = c;
                if (n < q.M) c *= bl / n;
            }
        }
        ++i;
    }
    return true;
}

/* V *= eps t^{-1 + B eps} (its variable outside Y) or 1/B - eps t^{-1 + B eps} (inside Y) for a series V that starts at
   eps^z; a: the variable's series */
template <int MAXM>
DEV void subset_factor(double (&V)[MAXM + 1], int z, const double *a, bool inY, int M) {
#pragma unroll
    for (int n = MAXM; n >= 0; --n) {
        if (n > M) continue;
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k <= n; ++k) {
            if (k < z || (k == n && !inY)) continue;
            const double f = k == n ? a[0] : (inY ? -a[n - k] : a[n - k]);
            acc = fma(V[k], f, acc);
        }
        V[n] = acc;
    }
}

/* Undeformed sectors: sum over Y of G_Y(eps) V_Y(eps), V_Y the product of the variables' factors.  The products over all
   but the last of the (at most four) variables are made once per point, 2^(sigma - 1) series in local memory.
   This regrouped sum keeps the rounding of a product of the same factors in the same order for every Y: near the faces
   t_j = 0 the terms cancel, and what is left there of their rounding is all of the error of a four-pole sector's sum.
   Bound by the FP64 pipe.  With the series and their products hoisted out of the subset loop, no arithmetic on zero
   imaginary parts or zero coefficients, and no logarithm where the order does not ask for it, the FP64 passes (16
   shifts) went from 32.2 to 16.2 ms (four-pole double box, n = 8191) and, with 8 shifts, from 5.36 to 2.88 ms (massless
   box, n = 65521).  The sum over the subsets rounds as it did with every step in the loop; the weight, one product of all
   x (1 - x) (weight64), in its last digit otherwise. */
template <int S, bool DEF, int MAXM, class Pol>
DEV typename EnableIf<!DEF>::type point_integrand(const PackedSector &s, const Pol &P, const double *x, int r, double,
                                                  const Exps &ex, cd (&out)[MAXM + 1], uint32_t &) {
#pragma unroll
    for (int n = 0; n <= MAXM; ++n) out[n] = mk(0.0, 0.0);
    const Subsets q{s.sigma, s.M, (unsigned)s.sing_mask};
    double t[S], tm[S], Lt[S], a[S][MAXM + 1], w;
    if (!point_setup<S, MAXM>(s, x, r, q, t, tm, Lt, a, w)) return;
    constexpr int NPRE = S < 4 ? S : 4; /* variables in the shared products: sigma - 1, at most NPRE - 1 */
    double pre[1 << (NPRE - 1)][MAXM + 1];
    const int np = q.sigma < NPRE ? (q.sigma > 0 ? q.sigma - 1 : 0) : NPRE - 1;
#pragma unroll
    for (int n = 0; n <= MAXM; ++n) pre[0][n] = n == 0 ? 1.0 : 0.0;
    for (int i = 0; i < np; ++i)
        for (int k = 0; k < (1 << i); ++k) {
            double V[MAXM + 1], W[MAXM + 1];
#pragma unroll
            for (int n = 0; n <= MAXM; ++n) V[n] = W[n] = pre[k][n];
            const int z = i - __popc(k);
            subset_factor<MAXM>(V, z, a[i], false, q.M);
            subset_factor<MAXM>(W, z, a[i], true, q.M);
#pragma unroll
            for (int n = 0; n <= MAXM; ++n) {
                pre[k][n] = V[n];
                pre[k + (1 << i)][n] = W[n];
            }
        }
    double o[MAXM + 1];
#pragma unroll
    for (int n = 0; n <= MAXM; ++n) o[n] = 0.0;
    unsigned Y = 0, count = 0;
    do {
        double tt[S];
#pragma unroll
        for (int j = 0; j < S; ++j) tt[j] = (Y >> j) & 1u ? 0.0 : t[j];
        const int need = q.need(count);
        double g, X;
        eval_G<S>(s, P, Y, tt, Lt, MAXM > 0 && need > 0, ex, g, X);
        double V[MAXM + 1];
        const unsigned low = count & ((1u << np) - 1u);
#pragma unroll
        for (int n = 0; n <= MAXM; ++n) V[n] = pre[low][n];
        int z = np - __popc(low);
        for (int i = np; i < q.sigma; ++i) {
            const bool inY = (count >> i) & 1u;
            subset_factor<MAXM>(V, z, a[i], inY, q.M);
            z += inY ? 0 : 1;
        }
#pragma unroll
        for (int n = 0; n <= MAXM; ++n) {
            if (n > need) break;
#pragma unroll
            for (int k = 0; k + n <= MAXM; ++k)
                if (k >= z && n + k <= q.M) o[n + k] = fma(g, V[k], o[n + k]);
            if (n < need) {
                g = g * X;
                if (n > 0) g *= 1.0 / (n + 1);
            }
        }
        ++count;
        Y = (Y - q.smask) & q.smask;
    } while (Y != 0);
#pragma unroll
    for (int n = 0; n <= MAXM; ++n) out[n].x = o[n] * w;
}

/* Deformed sectors (at most two poles in the physical integrals): the subsets are enumerated like a binary counter, and
   whenever both halves of a bit are done (variable i not zeroed, zeroed) they are combined to
   a_i (G - G0) + G0 / B_i, so that at most sigma complex series wait, on a stack in local memory. */
template <int S, bool DEF, int MAXM, class Pol>
DEV typename EnableIf<DEF>::type point_integrand(const PackedSector &s, const Pol &P, const double *x, int r, double lam,
                                                 const Exps &ex, cd (&out)[MAXM + 1], uint32_t &fails) {
#pragma unroll
    for (int n = 0; n <= MAXM; ++n) out[n] = mk(0.0, 0.0);
    const Subsets q{s.sigma, s.M, (unsigned)s.sing_mask};
    double t[S], tm[S], Lt[S], a[S][MAXM + 1], w;
    if (!point_setup<S, MAXM>(s, x, r, q, t, tm, Lt, a, w)) return;
    cd st[S][MAXM + 1], cur[MAXM + 1];
    int sp = 0;
    unsigned Y = 0, count = 0;
    for (;;) {
        double tt[S], ttm[S];
#pragma unroll
        for (int j = 0; j < S; ++j) {
            const bool zj = (Y >> j) & 1u;
            tt[j] = zj ? 0.0 : t[j];
            ttm[j] = zj ? 1.0 : tm[j];
        }
        const int need = q.need(count);
        cd X;
        eval_G<S>(s, P, Y, tt, ttm, Lt, lam, MAXM > 0 && need > 0, ex, cur[0], X, fails);
#pragma unroll
        for (int n = 1; n <= MAXM; ++n) {
            if (n > need) break;
            cur[n] = cmul(cur[n - 1], X);
            if (n > 1) cur[n] = cscale(cur[n], 1.0 / n);
        }
        int i = 0;
        for (unsigned b = count; b & 1u; b >>= 1, ++i) {
            --sp;
            /* the combined series is needed to this order; its lower half, which a_i raises by one, to one less */
            const int m = q.M - q.sigma + (i + 1) + __popc(b >> 1);
            cd d[MAXM + 1];
#pragma unroll
            for (int n = 0; n < MAXM; ++n) {
                if (n >= m) break;
                d[n] = csub(st[sp][n], cur[n]);
            }
#pragma unroll
            for (int n = 0; n <= MAXM; ++n) {
                if (n > m) break;
                cd acc = cscale(cur[n], a[i][0]);
#pragma unroll
                for (int k = 1; k <= n; ++k) acc = mk(fma(a[i][k], d[n - k].x, acc.x), fma(a[i][k], d[n - k].y, acc.y));
                cur[n] = acc;
            }
        }
        ++count;
        Y = (Y - q.smask) & q.smask;
        if (Y == 0) break;
#pragma unroll
        for (int n = 0; n <= MAXM; ++n) st[sp][n] = cur[n];
        ++sp;
    }
#pragma unroll
    for (int n = 0; n <= MAXM; ++n)
        if (n <= q.M) out[n] = cscale(cur[n], w);
}

/* ------------------------------------------------------------------ staging a sector into shared memory */
DEV void stage_sector(const unsigned char *packed, int64_t sectors_off, int64_t terms_off, int psec,
                      unsigned char *smem) {
    const PackedSector *ps = reinterpret_cast<const PackedSector *>(packed + sectors_off) + psec;
    const int4 *src = reinterpret_cast<const int4 *>(ps);
    int4 *dst = reinterpret_cast<int4 *>(smem);
    constexpr int NS = (int)(sizeof(PackedSector) / 16);
    for (int k = threadIdx.x; k < NS; k += blockDim.x) dst[k] = src[k];
    if (threadIdx.x < 8) {
        const double B = (double)ps->B[threadIdx.x];
        qmc_sec.B[threadIdx.x] = B;
        qmc_sec.rB[threadIdx.x] = 1.0 / B; /* used for singular variables only: B != 0 there */
    }
    const int nt = ps->n_terms;
    const int4 *tsrc = reinterpret_cast<const int4 *>(packed + terms_off) + ps->term0;
    int4 *tdst = dst + NS;
    for (int k = threadIdx.x; k < nt; k += blockDim.x) tdst[k] = tsrc[k];
}

/* Smallest integer r with fma(r, 1/n, delta) >= 1: the lattice point x = {r/n + delta} wraps exactly for
   r >= R, so the per-point wrap test is an integer compare (evaluated once per item and shift). */
DEV uint32_t wrap_threshold(double delta, uint32_t n, double invn) {
    double g = ceil((1.0 - delta) * (double)n);
    uint32_t R = g <= 0.0 ? 0u : (g >= (double)n ? n : (uint32_t)g);
    while (R > 0 && fma((double)(R - 1), invn, delta) >= 1.0) --R;
    while (R < n && fma((double)R, invn, delta) < 1.0) ++R;
    return R;
}

/* ------------------------------------------------------------------ FP64 islands of a mixed pass
 * The subtraction of Eq. 11 cancels near the faces t_j = 0 of the singular variables (the remark after Eq. 12),
 * and that is where FP32 loses the digits a sector's error budget needs.  A mixed pass may evaluate a sector in
 * FP32 except at its island points, which the FP64 kernel evaluates: at level L, the points whose product over
 * the singular variables of (k_j + 1) / n is below 10^-(L+1), k_j = floor(n x_j) the integer part of the shifted
 * lattice coordinate (x_j = (k_j + b_j) / n, 0 <= b_j < 1).  The FP32 kernels, the FP64 kernel and the probe take
 * this decision with the functions below alone -- integer steps and correctly rounded FP32 operations -- so
 * every kernel sees the same islands. */
DEV uint32_t shift_floor(double delta, uint32_t n) {
    const double fl = floor(__dmul_rn(delta, (double)n));
    return fl >= (double)n ? n - 1u : (uint32_t)fl;
}

DEV uint32_t shifted_index(uint32_t r, uint32_t a, uint32_t n) {
    const uint32_t k = r + a;
    return k >= n ? k - n : k;
}

DEV float island_rn(uint32_t n) { return __frcp_rn(__uint2float_rn(n)); }

/* prod over the singular variables (mask) of (k_j + 1) / n, floored at 1e-30 after each factor (no subnormals) */
template <int S>
DEV float island_key(const uint32_t (&k)[S], unsigned mask, float rn) {
    float c = 1.f;
#pragma unroll
    for (int j = 0; j < S; ++j)
        if ((mask >> j) & 1u) c = fmaxf(__fmul_rn(c, __fmul_rn(__uint2float_rn(k[j] + 1u), rn)), 1e-30f);
    return c;
}

/* the threshold of level L: 10^-(L+1) rounded to FP32 */
DEV float island_xi(int L) {
    return L == 0 ? 1e-1f : L == 1 ? 1e-2f : L == 2 ? 1e-3f : L == 3 ? 1e-4f : L == 4 ? 1e-5f : 1e-6f;
}

/* the number of levels a point with this key is an island at */
DEV int island_bin(float key) {
    int b = 0;
#pragma unroll
    for (int L = 0; L < QMC_ISLAND_LEVELS; ++L) b += key < island_xi(L) ? 1 : 0;
    return b;
}

/* island level of a sector precision code of a mixed pass (2 + L), or -1 */
DEV int island_level(int code) { return code >= 2 && code < 2 + QMC_ISLAND_LEVELS ? code - 2 : -1; }

DEV void kahan_add(double &s, double &c, double v) {
    const double y = v - c;
    const double t = s + y;
    c = (t - s) - y;
    s = t;
}

/* ------------------------------------------------------------------ job lookup */
/* the job whose item range contains `item` (jobs are in increasing item_begin) */
DEV int find_job(const JobTable &jt, long long item) {
    int lo = 0, hi = jt.n_jobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jt.jobs[mid].item_begin <= item) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

/* nonzero once the job's abort flag (device-visible, e.g. mapped pinned host memory) is set */
DEV int job_aborted(const Job &J) { return J.abort ? *J.abort : 0; }

/* ------------------------------------------------------------------ K1: persistent FP64 evaluation */
template <int S, int MAXM>
__device__ __noinline__ void point_integrand_taylor(const PackedSector &s, const PackedTerm *T, const double *x, int r,
                                                    Exps ex, double *out);

/* TAYLOR: the sectors of class 2 (endpoint exponents alpha <= -2), evaluated by point_integrand_taylor */
template <int S, bool DEF, int MAXM, class Pol, bool TAYLOR = false>
DEV void eval_f64_body(const JobTable &jt) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long s_item;
    __shared__ int s_job, s_abort;
    __shared__ double s_red[16][2 * (MAXM + 1)];
    __shared__ uint32_t s_fail[16];
    /* per warp: lattice residues r_j of the points gathered for evaluation (at most 63 wait between batches) */
    __shared__ uint32_t s_queue[8][64 * S];
    const PackedSector &sec = *reinterpret_cast<const PackedSector *>(smem);
    const PackedTerm *T = reinterpret_cast<const PackedTerm *>(smem + sizeof(PackedSector));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    uint32_t *queue = s_queue[warp & 7];
    int cur = -1, cur_job = -1;
    logtab_init(); /* made visible by the __syncthreads() after the first item fetch */
    for (;;) {
        if (threadIdx.x == 0) {
            const long long it = (long long)atomicAdd(jt.counter, 1ull);
            s_item = it;
            s_job = it < jt.total_items ? find_job(jt, it) : 0;
            s_abort = it < jt.total_items ? job_aborted(jt.jobs[s_job]) : 0;
        }
        __syncthreads();
        const long long item = s_item;
        if (item >= jt.total_items) break;
        const int jb = s_job;
        const Job &J = jt.jobs[jb];
        const long long local = item - J.item_begin;
        if (s_abort) { /* the pass was stopped: its remaining items contribute nothing */
            if ((int)threadIdx.x < J.n_slots * 2) J.partials[local * J.n_slots * 2 + threadIdx.x] = 0.0;
            if (threadIdx.x == 0) J.part_fails[local] = 0;
            __syncthreads();
            continue;
        }
        const long long per_sector = (long long)J.m * J.chunks;
        const int ls = (int)(local / per_sector);
        const long long rem = local - (long long)ls * per_sector;
        const int shift = (int)(rem / J.chunks);
        const long long chunk = rem - (long long)shift * J.chunks;
        const int psec = J.sector_begin + ls;
        int level = -1; /* island level: this kernel evaluates only the sector's island points */
        if (J.sector_prec) {
            /* mixed pass: items of sectors evaluated in FP32 belong to the other kernel; of sectors with FP64
               islands, this kernel takes the islands and writes the item's partial first (it launches first) */
            const PackedSector *gps = reinterpret_cast<const PackedSector *>(J.packed + J.sectors_off) + psec;
            const int code = J.sector_prec[gps->orig_index];
            if (code == 1) {
                __syncthreads();
                continue;
            }
            level = island_level(code);
        }
        if (psec != cur || jb != cur_job) {
            stage_sector(J.packed, J.sectors_off, J.terms_off, psec, smem);
            __syncthreads();
            cur = psec;
            cur_job = jb;
        }
        const Exps ex = Pol::exps(J);
        const Pol pol = Pol::make(T, sec, psec);
        const uint32_t n = J.n;
        const double invn = J.invn;
        const double lam = J.lambda[sec.orig_index];
        double delta[S];
        uint32_t rj[S], Rj[S], zs[S], aj[S];
        const long long i0 = chunk * (long long)blockDim.x * jt.P + threadIdx.x;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            delta[j] = J.shifts[6 * shift + j];
            rj[j] = (uint32_t)(((unsigned long long)i0 * J.z[j]) % n);
            Rj[j] = wrap_threshold(delta[j], n, invn);
            zs[j] = J.zstep[j];
            aj[j] = shift_floor(delta[j], n);
        }
        const float rn = island_rn(n), xi = island_xi(level < 0 ? 0 : level);
        const unsigned smask = (unsigned)sec.sing_mask;
        /* a thread sums its points plainly; the block combines threads by a shuffle tree, warps and items
           with compensated (Kahan) sums */
        double acc[2 * (MAXM + 1)];
#pragma unroll
        for (int q = 0; q < 2 * (MAXM + 1); ++q) acc[q] = 0.0;
        uint32_t fails = 0;
        /* The warp gathers its points (every point, or the islands) into its queue 32 lanes at a time and
           evaluates them in batches of 32, so island points keep whole warps busy.  With every point taken,
           lane l evaluates its own points in order, as a plain loop would. */
        int qn = 0, p = 0;
        for (;;) {
            while (qn < 32 && p < jt.P) {
                const long long i = i0 + (long long)p * blockDim.x;
                bool take = i < (long long)n;
                if (take && level >= 0) {
                    uint32_t k[S];
#pragma unroll
                    for (int j = 0; j < S; ++j) k[j] = shifted_index(rj[j], aj[j], n);
                    take = island_key<S>(k, smask, rn) < xi;
                }
                const unsigned bal = __ballot_sync(0xffffffffu, take);
                if (take) {
                    const int pos = qn + __popc(bal & ((1u << lane) - 1u));
#pragma unroll
                    for (int j = 0; j < S; ++j) queue[pos * S + j] = rj[j];
                }
                qn += __popc(bal);
#pragma unroll
                for (int j = 0; j < S; ++j) {
                    const uint32_t v = rj[j] + zs[j];
                    rj[j] = v >= n ? v - n : v;
                }
                ++p;
            }
            if (qn == 0) break;
            __syncwarp();
            if (lane < qn) {
                double x[S];
#pragma unroll
                for (int j = 0; j < S; ++j) {
                    const uint32_t r = queue[lane * S + j];
                    x[j] = fma((double)r, invn, delta[j]) - (r >= Rj[j] ? 1.0 : 0.0);
                }
                cd val[MAXM + 1];
                if constexpr (TAYLOR) {
                    double v[MAXM + 1];
                    point_integrand_taylor<S, MAXM>(sec, T, x, jt.r, ex, v);
#pragma unroll
                    for (int m = 0; m <= MAXM; ++m) val[m] = mk(v[m], 0.0);
                } else {
                    point_integrand<S, DEF, MAXM>(sec, pol, x, jt.r, lam, ex, val, fails);
                }
#pragma unroll
                for (int m = 0; m <= MAXM; ++m) {
                    acc[2 * m] += val[m].x;
                    acc[2 * m + 1] += val[m].y;
                }
            }
            __syncwarp();
            const int rest = qn > 32 ? qn - 32 : 0;
            if (lane < rest) {
#pragma unroll
                for (int j = 0; j < S; ++j) queue[lane * S + j] = queue[(32 + lane) * S + j];
            }
            __syncwarp();
            qn = rest;
        }
#pragma unroll
        for (int q = 0; q < 2 * (MAXM + 1); ++q) {
            double v = acc[q];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
            if (lane == 0) s_red[warp][q] = v;
        }
        uint32_t f = fails;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) f += __shfl_down_sync(0xffffffffu, f, off);
        if (lane == 0) s_fail[warp] = f;
        __syncthreads();
        if (threadIdx.x < 32) {
            const int q = threadIdx.x;
            if (q < J.n_slots * 2) {
                double s2 = 0.0, c2 = 0.0;
                if (q < 2 * (MAXM + 1))
                    for (int w = 0; w < nwarps; ++w) kahan_add(s2, c2, s_red[w][q]);
                J.partials[local * J.n_slots * 2 + q] = s2 - c2;
            }
            if (q == 0) {
                uint32_t tf = 0;
                for (int w = 0; w < nwarps; ++w) tf += s_fail[w];
                J.part_fails[local] = tf;
            }
        }
        __syncthreads();
    }
}

template <int S, bool DEF, int MAXM>
__global__ void __launch_bounds__(256) qmc_eval_kernel(const __grid_constant__ JobTable jt) {
    eval_f64_body<S, DEF, MAXM, TabPol<S>>(jt);
}

/* ================================================================== endpoint exponents alpha <= -2 (class 2)
 * Sec. II, Eq. (11) with p > 0: for a variable with t^{a + b eps}, a = -1 - p,
 *   int_0^1 t^{a+b eps} f(t) dt = int_0^1 t^{a+b eps} [f(t) - sum_{k<=p} f^(k)(0) t^k/k!] dt
 *                                 + sum_{k<=p} f^(k)(0) / (k! (a + k + 1 + b eps)),
 * applied to every variable with alpha_j <= -1 of the sector (the operators of different variables commute).
 * Per point each such variable takes one of three roles: its value (factor t^{a+b eps}), a subtracted Taylor term,
 * or a pole term.  The Taylor coefficients of f in the variables set to zero (the subset Z) are the coefficients of
 * truncated power series ("jets"): the jets of U~ and F~ restricted to those variables, raised to their
 * eps-dependent powers by the power recurrence of a series, P0 |k| R_k = sum_{0<l<=k} (a |l| - |k-l|) P_l R_{k-l}
 * (from P E R = a R E P with the Euler operator E), and multiplied.  The remainder of a variable with
 * t_j < QMC_TAYLOR_SMALL_T is taken from its own series (orders p_j < k <= p_j + QMC_TAYLOR_EXTRA), because the
 * difference loses its digits there.  Undeformed sectors only (F~ of one sign); FP64, table evaluator. */
#define QMC_TAYLOR_JET (QMC_TAYLOR_Q * QMC_TAYLOR_Q)

/* c = a * b for eps series of length L (truncated) */
template <int L>
DEV void ser_mul(const double *a, const double *b, double *c, int n) {
    for (int i = n - 1; i >= 0; --i) {
        double s = 0.0;
        for (int k = 0; k <= i; ++k) s = fma(a[k], b[i - k], s);
        c[i] = s;
    }
}

/* exp(x eps) t^A as a series: t^A x^m / m! */
template <int L>
DEV void ser_power_exp(double tA, double x, double *out, int n) {
    double c = tA;
    for (int m = 0; m < n; ++m) {
        out[m] = c;
        c = c * x / (m + 1);
    }
}

/* R = P^{a0 + a1 eps} for a jet P over d0 x d1 orders (row-major, P[0] > 0); R holds L-term series per entry */
template <int L>
DEV void jet_power(const double *P, int d0, int d1, int a0, int a1, double *R, int n) {
    const double P0 = P[0];
    ser_power_exp<L>(ipow(P0, a0), (double)a1 * qlog(P0), R, n);
    const double inv0 = 1.0 / P0;
    for (int k0 = 0; k0 < d0; ++k0)
        for (int k1 = 0; k1 < d1; ++k1) {
            const int kk = k0 + k1;
            if (kk == 0) continue;
            double acc[L];
            for (int m = 0; m < n; ++m) acc[m] = 0.0;
            for (int l0 = 0; l0 <= k0; ++l0)
                for (int l1 = 0; l1 <= k1; ++l1) {
                    const int ll = l0 + l1;
                    if (ll == 0) continue;
                    const double p = P[l0 * d1 + l1];
                    if (p == 0.0) continue;
                    const double *r = R + ((k0 - l0) * d1 + (k1 - l1)) * L;
                    const double c0 = p * (double)(a0 * ll - (kk - ll)), c1 = p * (double)(a1 * ll);
                    for (int m = n - 1; m >= 0; --m) acc[m] = fma(c0, r[m], m > 0 ? fma(c1, r[m - 1], acc[m]) : acc[m]);
                }
            double *Rk = R + (k0 * d1 + k1) * L;
            const double s = inv0 / (double)kk;
            for (int m = 0; m < n; ++m) Rk[m] = acc[m] * s;
        }
}

/* w(x) * (sector integrand) at x for a class-2 sector, slots 0..M (slot n = coefficient of eps^(n - sigma)) */
template <int S, int MAXM>
__device__ __noinline__ void point_integrand_taylor(const PackedSector &s, const PackedTerm *T, const double *x, int r,
                                                    Exps ex, double *out) {
    constexpr int L = MAXM + 1;
    const int n = s.M + 1;
    for (int m = 0; m < L; ++m) out[m] = 0.0;
    double t[S], lt[S], w = 1.0;
    for (int j = 0; j < S; ++j) {
        double tm, wj;
        if (!(x[j] > 0.0)) return; /* the weight vanishes at x = 0 */
        transform(r, x[j], t[j], tm, wj);
        w *= wj;
        lt[j] = qlog(t[j]);
    }
    int sv[QMC_TAYLOR_MAX_Z], pv[QMC_TAYLOR_MAX_Z];
    bool small[QMC_TAYLOR_MAX_Z];
    int sigma = 0;
    double base[L];
    for (int m = 0; m < L; ++m) base[m] = 0.0;
    base[0] = s.D;
    for (int j = 0; j < S; ++j) {
        if (s.A[j] <= -1) {
            sv[sigma] = j;
            pv[sigma] = -s.A[j] - 1;
            small[sigma] = t[j] < QMC_TAYLOR_SMALL_T;
            ++sigma;
        } else if (s.A[j] != 0 || s.B[j] != 0) {
            double f[L];
            ser_power_exp<L>(ipow(t[j], s.A[j]), (double)s.B[j] * lt[j], f, n);
            ser_mul<L>(base, f, base, n);
        }
    }
    double tpow[QMC_TAYLOR_MAX_Z][L];
    for (int i = 0; i < sigma; ++i) {
        const int j = sv[i];
        ser_power_exp<L>(ipow(t[j], s.A[j]), (double)s.B[j] * lt[j], tpow[i], n);
    }
    const double sgnF = s.kind == 1 ? -1.0 : 1.0; /* F~ < 0 everywhere: |F~| here, the phase on the host */
    double PU[QMC_TAYLOR_JET], PF[QMC_TAYLOR_JET];
    double RU[QMC_TAYLOR_JET * L], RF[QMC_TAYLOR_JET * L];
    for (unsigned zm = 0; zm < (1u << sigma); ++zm) {
        int zi[QMC_TAYLOR_MAX_Z], q[QMC_TAYLOR_MAX_Z], nz = 0;
        for (int i = 0; i < sigma; ++i)
            if ((zm >> i) & 1u) {
                zi[nz] = i;
                q[nz] = small[i] ? pv[i] + QMC_TAYLOR_EXTRA : pv[i];
                ++nz;
            }
        /* the values of the variables outside Z: their remainder as a difference, so zero where it is small */
        double pre[L];
        for (int m = 0; m < L; ++m) pre[m] = base[m];
        bool dead = false;
        for (int i = 0; i < sigma; ++i)
            if (!((zm >> i) & 1u)) {
                if (small[i]) dead = true;
                else ser_mul<L>(pre, tpow[i], pre, n);
            }
        if (dead) continue;
        const int d0 = nz >= 1 ? q[0] + 1 : 1, d1 = nz == 2 ? q[1] + 1 : 1;
        const int nj = d0 * d1;
        for (int k = 0; k < nj; ++k) PU[k] = PF[k] = 0.0;
        for (int a = 0; a < s.nU + s.nF; ++a) {
            const PackedTerm &tm = T[a];
            const int k0 = nz >= 1 ? tm.e[sv[zi[0]]] : 0, k1 = nz == 2 ? tm.e[sv[zi[1]]] : 0;
            if (k0 >= d0 || k1 >= d1) continue;
            double v = a < s.nU ? tm.c : sgnF * tm.c;
            for (int j = 0; j < S; ++j) {
                bool inZ = false;
                for (int i = 0; i < nz; ++i) inZ |= sv[zi[i]] == j;
                if (!inZ) v *= ipow(t[j], tm.e[j]);
            }
            (a < s.nU ? PU : PF)[k0 * d1 + k1] += v;
        }
        jet_power<L>(PU, d0, d1, ex.eU0, ex.eU1, RU, n);
        jet_power<L>(PF, d0, d1, -ex.eF0, -ex.eF1, RF, n);
        /* roles: every subset of Z takes the pole role, the rest of Z the subtracted one */
        for (unsigned tmk = 0; tmk < (1u << nz); ++tmk)
            for (int k0 = 0; k0 < d0; ++k0)
                for (int k1 = 0; k1 < d1; ++k1) {
                    const int kk[2] = {k0, k1};
                    bool skip = false;
                    for (int i = 0; i < nz; ++i) {
                        const int vi = zi[i];
                        const bool pole = (tmk >> i) & 1u;
                        if (pole && kk[i] > pv[vi]) skip = true;
                        /* subtracted: Taylor terms k <= p where the remainder is a difference, series terms
                           k > p where it comes from its series */
                        if (!pole && ((kk[i] <= pv[vi]) == small[vi])) skip = true;
                    }
                    if (skip) continue;
                    double g[L];
                    for (int m = 0; m < L; ++m) g[m] = 0.0;
                    for (int l0 = 0; l0 <= k0; ++l0)
                        for (int l1 = 0; l1 <= k1; ++l1) {
                            double pr[L];
                            ser_mul<L>(RU + (l0 * d1 + l1) * L, RF + ((k0 - l0) * d1 + (k1 - l1)) * L, pr, n);
                            for (int m = 0; m < n; ++m) g[m] += pr[m];
                        }
                    double term[L];
                    ser_mul<L>(pre, g, term, n);
                    int shift = 0;
                    for (int i = 0; i < nz; ++i) {
                        const int vi = zi[i], j = sv[vi];
                        if ((tmk >> i) & 1u) {
                            const int c = s.A[j] + kk[i] + 1;
                            if (c == 0) {
                                for (int m = 0; m < n; ++m) term[m] /= (double)s.B[j];
                                ++shift;
                            } else {
                                double sr[L], f = 1.0 / c;
                                const double ratio = -(double)s.B[j] / c;
                                for (int m = 0; m < n; ++m) {
                                    sr[m] = f;
                                    f *= ratio;
                                }
                                ser_mul<L>(term, sr, term, n);
                            }
                        } else {
                            const double sg = kk[i] <= pv[vi] ? -1.0 : 1.0;
                            double f[L];
                            const double tk = sg * ipow(t[j], kk[i]);
                            for (int m = 0; m < n; ++m) f[m] = tk * tpow[vi][m];
                            ser_mul<L>(term, f, term, n);
                        }
                    }
                    const int lo = sigma - shift;
                    for (int m = lo; m < n; ++m) out[m] += term[m - lo];
                }
    }
    for (int m = 0; m < n; ++m) out[m] *= w;
}

template <int S, int MAXM>
__global__ void __launch_bounds__(256) qmc_eval_kernel_taylor(const __grid_constant__ JobTable jt) {
    eval_f64_body<S, false, MAXM, TabPol<S>, true>(jt);
}

/* ================================================================== FP32 path of the mixed-precision pass
 * The integrand is evaluated in FP32: GB300 issues ~58x more FP32 than FP64 operations.  What stays exact or
 * FP64: the lattice index arithmetic (integers), 1 - x (formed from integers, never by subtraction), the
 * accumulation of the point values (double-float per thread, FP64 per work item and across items). */
struct cf {
    float x, y;
};
DEV cf mkf(float x, float y) { return cf{x, y}; }
/* Complex FP32 arithmetic on GB300's packed two-lane FP32 instructions (one instruction for the real and the
   imaginary part); each lane rounds exactly like the scalar form (x*y + z with one rounding, products rounded
   before they are added). */
DEV float2 f2_(cf a) { return make_float2(a.x, a.y); }
DEV cf cf_(float2 a) { return cf{a.x, a.y}; }
DEV cf caddf(cf a, cf b) { return cf_(__fadd2_rn(f2_(a), f2_(b))); }
DEV cf csubf(cf a, cf b) { return cf_(__fadd2_rn(f2_(a), make_float2(-b.x, -b.y))); }
DEV cf cscalef(cf a, float s) { return cf_(__fmul2_rn(f2_(a), make_float2(s, s))); }
/* (a.x b.x - a.y b.y, a.x b.y + a.y b.x) = (a.x, a.x) * (b.x, b.y) + rn((-a.y, a.y) * (b.y, b.x)) */
DEV cf cmulf(cf a, cf b) {
    return cf_(__ffma2_rn(make_float2(a.x, a.x), f2_(b), __fmul2_rn(make_float2(-a.y, a.y), make_float2(b.y, b.x))));
}
/* a + (c_hi + c_lo) m for a real coefficient split in two floats and a complex monomial m */
DEV cf cfma2f(float hi, float lo, cf m, cf a) {
    return cf_(__ffma2_rn(make_float2(hi, hi), f2_(m), __ffma2_rn(make_float2(lo, lo), f2_(m), f2_(a))));
}
/* the reciprocal of the squared modulus from the fast approximate division (2 ulp): the FP32 path's error is set by
   its rounding of products and sums, and an IEEE-rounded reciprocal costs several instructions more */
DEV cf cinvf(cf a) {
    const float d = __fdividef(1.f, fmaf(a.x, a.x, a.y * a.y));
    return cf{a.x * d, -a.y * d};
}
DEV cf cipowf(cf z, int e) {
    cf r = mkf(1.f, 0.f);
    int k = e < 0 ? -e : e;
    for (int i = 0; i < k; ++i) r = cmulf(r, z);
    return e < 0 ? cinvf(r) : r;
}
DEV float ipowf_(float v, int e) {
    float r = 1.f;
    int k = e < 0 ? -e : e;
    for (int i = 0; i < k; ++i) r *= v;
    return e < 0 ? __frcp_rn(r) : r;
}
DEV cf clogf_p(cf z) { return cf{0.5f * __logf(fmaf(z.x, z.x, z.y * z.y)), atan2f(z.y, z.x)}; }
DEV float arg_mi0f(float x, float y) { return (y == 0.f) ? (x < 0.f ? -3.14159265358979f : 0.f) : atan2f(y, x); }
DEV cf clogf_mi0(cf z) { return cf{0.5f * __logf(fmaf(z.x, z.x, z.y * z.y)), arg_mi0f(z.x, z.y)}; }

DEV float phi_poly_f(int r, float x) {
    switch (r) {
        case 0: return x;
        case 1: return x * x * fmaf(-2.f, x, 3.f);
        case 2: return x * x * x * fmaf(x, fmaf(6.f, x, -15.f), 10.f);
        default: {
            const float x2 = x * x;
            return x2 * x2 * fmaf(x, fmaf(x, fmaf(-20.f, x, 70.f), -84.f), 35.f);
        }
    }
}
/* x and y = 1 - x are both given (each accurate relative to itself) */
DEV void transform_f(int r, float x, float y, float &t, float &tm, float &w) {
    const bool lo = x <= y;
    const float p = phi_poly_f(r, lo ? x : y);
    const float q = 1.f - p;
    t = lo ? p : q;
    tm = lo ? q : p;
    const float xy = x * y;
    switch (r) {
        case 0: w = 1.f; break;
        case 1: w = 6.f * xy; break;
        case 2: w = 30.f * xy * xy; break;
        default: w = 140.f * xy * xy * xy; break;
    }
}

DEV uint64_t term_exps_f(const PackedTermF &T) { return *reinterpret_cast<const uint64_t *>(T.e); }

/* Term table of the FP32 path in shared memory (every lane of a warp reads the same term: a broadcast). */
struct SmemTabF {
    const PackedTermF *T;
    DEV float hi(int i) const { return T[i].hi; }
    DEV float lo(int i) const { return T[i].lo; }
    DEV uint64_t ex(int i) const { return term_exps_f(T[i]); }
};

/* coefficient as hi + lo float pair: two FMAs per term keep the coefficient exact to ~2^-48 */
template <int S, class Tab>
DEV float poly_rf(const Tab &T, int base, int n, const float *t) {
    float acc = 0.f;
    for (int a = base; a < base + n; ++a) {
        const uint64_t ew = T.ex(a);
        const float hi = T.hi(a), lo = T.lo(a);
        if (ew == 0) {
            acc += hi + lo;
            continue;
        }
        float m = 1.f;
        bool have = false;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            int e = (int)((ew >> (8 * j)) & 0xffu);
            if (e > 0) {
                if (!have) {
                    m = t[j];
                    have = true;
                    --e;
                }
                for (int k = 0; k < e; ++k) m *= t[j];
            }
        }
        acc = fmaf(hi, m, fmaf(lo, m, acc));
    }
    return acc;
}

template <int S, class Tab>
DEV cf poly_cf(const Tab &T, int base, int n, const cf *z) {
    cf acc = mkf(0.f, 0.f);
    for (int a = base; a < base + n; ++a) {
        const uint64_t ew = T.ex(a);
        const float hi = T.hi(a), lo = T.lo(a);
        if (ew == 0) {
            acc.x += hi + lo;
            continue;
        }
        cf m = mkf(1.f, 0.f);
        bool have = false;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            int e = (int)((ew >> (8 * j)) & 0xffu);
            if (e > 0) {
                if (!have) {
                    m = z[j];
                    have = true;
                    --e;
                }
                for (int k = 0; k < e; ++k) m = cmulf(m, z[j]);
            }
        }
        acc = cfma2f(hi, lo, m, acc);
    }
    return acc;
}

/* Polynomial evaluators of the FP32 path.  The integrand code below asks an evaluator for
     UFr(t, U, F)          U~ and F~ at real t (undeformed sectors, Eqs. 7-8),
     GH(t, g, h)           g_j = dF~/dt_j and h_p = d2F~/dt_j dt_k (p runs over j <= k, row-major upper
                           triangle) at real t, the inputs of the deformation of Eq. 14,
     UFc(z, needU, U, F)   U~ (1 when needU is false) and F~ at the deformed complex point z.
   TabPolF walks the staged term table and decodes each term's exponent bytes.  A generated evaluator
   (compiled at run time for one family of sector tables) holds every sector's monomials as straight-line code
   with shared sub-products and reads only the coefficients (hi + lo) from the same staged table. */
template <int S>
struct TabPolF {
    const PackedTermF *T;
    const PackedSector *s;
    DEV static TabPolF make(const PackedTermF *T, const PackedSector &s, int) { return TabPolF{T, &s}; }
    DEV static Exps exps(const Job &J) { return Exps{J.eU0, J.eU1, J.eF0, J.eF1}; }
    DEV void UFr(unsigned, const float *t, float &U, float &F) const {
        const SmemTabF tab{T};
        U = poly_rf<S>(tab, 0, s->nU, t);
        F = poly_rf<S>(tab, s->nU, s->nF, t);
    }
    DEV void GH(unsigned, const float *t, float *g, float *h) const {
        const SmemTabF tab{T};
        const int bG = s->nU + s->nF, bH = bG + s->nG;
#pragma unroll
        for (int j = 0; j < S; ++j) g[j] = poly_rf<S>(tab, bG + s->gstart[j], s->gstart[j + 1] - s->gstart[j], t);
#pragma unroll
        for (int p = 0; p < S * (S + 1) / 2; ++p)
            h[p] = poly_rf<S>(tab, bH + s->hstart[p], s->hstart[p + 1] - s->hstart[p], t);
    }
    DEV void UFc(unsigned, const cf *z, bool needU, cf &U, cf &F) const {
        const SmemTabF tab{T};
        U = needU ? poly_cf<S>(tab, 0, s->nU, z) : mkf(1.f, 0.f);
        F = poly_cf<S>(tab, s->nU, s->nF, z);
    }
};

template <int S>
DEV cf det_deform_f(const float (&A)[S][S], float lam) {
    if constexpr (S == 1) {
        return mkf(1.f, -lam * A[0][0]);
    } else if constexpr (S == 2) {
        const float tr = A[0][0] + A[1][1];
        const float dt = fmaf(A[0][0], A[1][1], -A[0][1] * A[1][0]);
        return mkf(fmaf(-lam * lam, dt, 1.f), -lam * tr);
    } else if constexpr (S == 3) {
        const float tr = A[0][0] + A[1][1] + A[2][2];
        const float e2 = fmaf(A[0][0], A[1][1], -A[0][1] * A[1][0]) + fmaf(A[0][0], A[2][2], -A[0][2] * A[2][0]) +
                         fmaf(A[1][1], A[2][2], -A[1][2] * A[2][1]);
        const float dt = A[0][0] * fmaf(A[1][1], A[2][2], -A[1][2] * A[2][1]) -
                         A[0][1] * fmaf(A[1][0], A[2][2], -A[1][2] * A[2][0]) +
                         A[0][2] * fmaf(A[1][0], A[2][1], -A[1][1] * A[2][0]);
        const float l2 = lam * lam;
        return mkf(fmaf(-l2, e2, 1.f), fmaf(l2 * lam, dt, -lam * tr));
    } else {
        cf J[S][S];
#pragma unroll
        for (int r = 0; r < S; ++r)
#pragma unroll
            for (int c = 0; c < S; ++c) J[r][c] = mkf(r == c ? 1.f : 0.f, -lam * A[r][c]);
        cf det = mkf(1.f, 0.f);
#pragma unroll
        for (int c = 0; c < S; ++c) {
            int p = c;
            float best = fabsf(J[c][c].x) + fabsf(J[c][c].y);
#pragma unroll
            for (int r = c + 1; r < S; ++r) {
                const float v = fabsf(J[r][c].x) + fabsf(J[r][c].y);
                if (v > best) {
                    best = v;
                    p = r;
                }
            }
            if (p != c) {
                det = cscalef(det, -1.f);
#pragma unroll
                for (int r = c + 1; r < S; ++r) {
                    if (r == p) {
#pragma unroll
                        for (int k = c; k < S; ++k) {
                            const cf tmp = J[c][k];
                            J[c][k] = J[r][k];
                            J[r][k] = tmp;
                        }
                    }
                }
            }
            det = cmulf(det, J[c][c]);
            const cf inv = cinvf(J[c][c]);
#pragma unroll
            for (int r = c + 1; r < S; ++r) {
                const cf f = cmulf(J[r][c], inv);
#pragma unroll
                for (int k = c + 1; k < S; ++k) J[r][k] = csubf(J[r][k], cmulf(f, J[c][k]));
            }
        }
        return det;
    }
}

/* det(I - i lam A) for S >= 4 in FP32, A = D + T H (D = diag((1-2t)g), T = diag(t(1-t)), H the Hessian of F):
   with s = T^(1/2), A is similar to the symmetric B = D + s H s, so the determinant is that of the complex
   symmetric N = I - i lam B, whose Hermitian part is the identity.  Gaussian elimination without pivoting is
   stable for matrices with a positive definite Hermitian part (every Schur complement keeps one, so no pivot
   vanishes); symmetric elimination works on the upper triangle only.  N holds the upper triangle row-major
   (S(S+1)/2 entries) and is overwritten. */
template <int S>
DEV cf det_sym_f(cf (&N)[S * (S + 1) / 2]) {
    auto at = [](int i, int j) { return i * S - i * (i - 1) / 2 + (j - i); }; /* i <= j */
    cf det = mkf(1.f, 0.f);
#pragma unroll
    for (int k = 0; k < S; ++k) {
        const cf dk = N[at(k, k)];
        det = cmulf(det, dk);
        if (k + 1 < S) {
            const cf inv = cinvf(dk);
#pragma unroll
            for (int i = k + 1; i < S; ++i) {
                const cf l = cmulf(N[at(k, i)], inv);
#pragma unroll
                for (int j = i; j < S; ++j) N[at(i, j)] = csubf(N[at(i, j)], cmulf(l, N[at(k, j)]));
            }
        }
    }
    return det;
}

/* FP32 sign check: rounding leaves |Im F| ~ 1e-7 |F| where the deformation vanishes; a point fails when
   Im F(z) exceeds that noise */
#define QMC_F32_SIGN_NOISE 4e-6f

template <int S, bool DEF, int MAXM, class Pol>
DEV void eval_G_f(const PackedSector &s, const Pol &P, unsigned Y, const float *tt, const float *ttm, const float *Lt,
                  float lam, int M, const Exps &ex, cf &G0, cf &X, uint32_t &fails) {
    const float D = s.Df;
    if constexpr (!DEF) {
        float U, F;
        P.UFr(Y, tt, U, F);
        if (s.kind == 1) F = -F;
        float g = D * ipowf_(U, ex.eU0) * ipowf_(F, -ex.eF0);
#pragma unroll
        for (int j = 0; j < S; ++j)
            for (int k = 0; k < s.A[j]; ++k) g *= tt[j];
        G0 = mkf(g, 0.f);
        X = mkf(0.f, 0.f);
        if (MAXM > 0 && M > 0) {
            float x = __logf(ipowf_(U, ex.eU1) * ipowf_(F, -ex.eF1));
#pragma unroll
            for (int j = 0; j < S; ++j)
                if (s.A[j] != -1 && s.B[j] != 0) x = fmaf((float)s.B[j], Lt[j], x);
            X = mkf(x, 0.f);
        }
    } else {
        float g[S], h[S * (S + 1) / 2];
        P.GH(Y, tt, g, h);
        cf detJ;
        if constexpr (S >= 4) {
            float s[S];
#pragma unroll
            for (int j = 0; j < S; ++j) {
                const float pj = tt[j] * ttm[j];
                s[j] = pj > 0.f ? pj * rsqrtf(pj) : 0.f;
            }
            cf N[S * (S + 1) / 2];
            int p = 0;
#pragma unroll
            for (int j = 0; j < S; ++j) {
#pragma unroll
                for (int k = j; k < S; ++k) {
                    const float b = (k == j) ? fmaf(ttm[j] - tt[j], g[j], tt[j] * ttm[j] * h[p]) : s[j] * s[k] * h[p];
                    N[p] = mkf(k == j ? 1.f : 0.f, -lam * b);
                    ++p;
                }
            }
            detJ = det_sym_f<S>(N);
        } else {
            float A[S][S];
            int p = 0;
#pragma unroll
            for (int j = 0; j < S; ++j) {
#pragma unroll
                for (int k = j; k < S; ++k) {
                    A[j][k] = tt[j] * ttm[j] * h[p];
                    if (k != j) A[k][j] = tt[k] * ttm[k] * h[p];
                    ++p;
                }
            }
#pragma unroll
            for (int j = 0; j < S; ++j) A[j][j] = fmaf(ttm[j] - tt[j], g[j], A[j][j]);
            detJ = det_deform_f<S>(A, lam);
        }
        cf z[S], q[S];
#pragma unroll
        for (int j = 0; j < S; ++j) {
            const float d = lam * ttm[j] * g[j];
            z[j] = mkf(tt[j], -tt[j] * d);
            q[j] = mkf(1.f, -d);
        }
        const bool needU = ex.eU0 != 0 || (MAXM > 0 && M > 0);
        cf U, F;
        P.UFc(Y, z, needU, U, F);
        fails += (F.y > QMC_F32_SIGN_NOISE * (fabsf(F.x) + fabsf(F.y))) ? 1u : 0u;
        cf G = cscalef(detJ, D);
        if (ex.eU0 != 0) G = cmulf(G, cipowf(U, ex.eU0));
        G = cmulf(G, cipowf(F, -ex.eF0));
        bool any_mono = false;
        float mono = 1.f;
#pragma unroll
        for (int j = 0; j < S; ++j)
            for (int k = 0; k < s.A[j]; ++k) {
                mono *= tt[j];
                any_mono = true;
            }
        if (any_mono) G = cscalef(G, mono);
#pragma unroll
        for (int j = 0; j < S; ++j)
            if (s.A[j] != 0) G = cmulf(G, cipowf(q[j], s.A[j]));
        G0 = G;
        X = mkf(0.f, 0.f);
        if (MAXM > 0 && M > 0) {
            cf x = csubf(cscalef(clogf_p(U), (float)ex.eU1), cscalef(clogf_mi0(F), (float)ex.eF1));
            /* log q_j with q_j = 1 - i d_j: (log(1 + d_j^2) / 2, -atan d_j) */
            float lr = 0.f;
#pragma unroll
            for (int j = 0; j < S; ++j) {
                if (s.B[j] != 0) {
                    const float Bj = (float)s.B[j];
                    if (s.A[j] != -1) x.x = fmaf(Bj, Lt[j], x.x);
                    const float d = -q[j].y;
                    lr = fmaf(Bj, __logf(fmaf(d, d, 1.f)), lr);
                    x.y = fmaf(-Bj, atanf(d), x.y);
                }
            }
            x.x = fmaf(0.5f, lr, x.x);
            X = x;
        }
    }
}

template <int S, bool DEF, int MAXM, class Pol>
DEV void point_integrand_f(const PackedSector &s, const Pol &P, const float *x, const float *y, int r, float lam,
                           const Exps &ex, cf (&out)[MAXM + 1], uint32_t &fails) {
    float t[S], tm[S], w = 1.f;
    bool bad = false;
#pragma unroll
    for (int j = 0; j < S; ++j) {
        float wj;
        transform_f(r, x[j], y[j], t[j], tm[j], wj);
        w *= wj;
        bad |= !(t[j] > 0.f) || !(tm[j] > 0.f);
    }
#pragma unroll
    for (int n = 0; n <= MAXM; ++n) out[n] = mkf(0.f, 0.f);
    if (bad || !(w > 0.f)) return;
    const int M = s.M;
    const unsigned smask = (unsigned)s.sing_mask;
    float Lt[S];
#pragma unroll
    for (int j = 0; j < S; ++j) Lt[j] = 0.f;
    if (MAXM > 0 && M > 0) {
#pragma unroll
        for (int j = 0; j < S; ++j)
            if (((smask >> j) & 1u) || s.B[j] != 0) Lt[j] = __logf(t[j]);
    }
    unsigned Y = 0;
    do {
        float tt[S], ttm[S];
#pragma unroll
        for (int j = 0; j < S; ++j) {
            const bool zj = (Y >> j) & 1u;
            tt[j] = zj ? 0.f : t[j];
            ttm[j] = zj ? 1.f : tm[j];
        }
        cf G0, X;
        eval_G_f<S, DEF, MAXM>(s, P, Y, tt, ttm, Lt, lam, M, ex, G0, X, fails);
        float V[MAXM + 1];
        V[0] = 1.f;
#pragma unroll
        for (int n = 1; n <= MAXM; ++n) V[n] = 0.f;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            if ((smask >> j) & 1u) {
                const bool inY = (Y >> j) & 1u;
                const float Bj = (float)s.B[j];
                float f[MAXM + 1];
                f[0] = inY ? __fdividef(1.f, Bj) : 0.f;
                float c = __fdividef(1.f, t[j]);
#pragma unroll
                for (int n = 1; n <= MAXM; ++n) {
                    f[n] = inY ? -c : c;
                    c *= Bj * Lt[j] / n;
                }
#pragma unroll
                for (int n = MAXM; n >= 0; --n) {
                    float acc = 0.f;
#pragma unroll
                    for (int k = 0; k <= n; ++k) acc = fmaf(V[k], f[n - k], acc);
                    V[n] = acc;
                }
            }
        }
        cf g = G0;
#pragma unroll
        for (int n = 0; n <= MAXM; ++n) {
            if (n <= M) {
#pragma unroll
                for (int k = 0; k + n <= MAXM; ++k)
                    if (n + k <= M) out[n + k] = caddf(out[n + k], cscalef(g, V[k]));
                g = cscalef(cmulf(g, X), 1.f / (n + 1));
            }
        }
        Y = (Y - smask) & smask;
    } while (Y != 0);
#pragma unroll
    for (int n = 0; n <= MAXM; ++n) out[n] = cscalef(out[n], w);
}

/* x = ((r + a) mod n + b)/n and 1 - x = ((n - 1 - (r + a) mod n) + (1 - b))/n, with delta * n = a + b */
DEV void lattice_f32(uint32_t r, uint32_t a, float b, uint32_t n, float invnf, float &x, float &y) {
    const uint32_t k = shifted_index(r, a, n);
    x = ((float)k + b) * invnf;
    y = ((float)(n - 1u - k) + (1.f - b)) * invnf;
}

DEV void split_shift(double delta, uint32_t n, uint32_t &a, float &b) {
    a = shift_floor(delta, n);
    b = (float)(__dmul_rn(delta, (double)n) - (double)a);
}

/* TwoSum: s + v = (s') + err exactly; the error goes into the compensation term */
DEV void two_sum_acc(float &s, float &c, float v) {
    const float t = s + v;
    const float bp = t - s;
    c += (s - (t - bp)) + (v - bp);
    s = t;
}

DEV void stage_sector_f(const unsigned char *packed, int64_t sectors_off, int64_t termsf_off, int psec,
                        unsigned char *smem) {
    const PackedSector *ps = reinterpret_cast<const PackedSector *>(packed + sectors_off) + psec;
    const int4 *src = reinterpret_cast<const int4 *>(ps);
    int4 *dst = reinterpret_cast<int4 *>(smem);
    constexpr int NS = (int)(sizeof(PackedSector) / 16);
    for (int k = threadIdx.x; k < NS; k += blockDim.x) dst[k] = src[k];
    const int nt = ps->n_terms;
    const int4 *tsrc = reinterpret_cast<const int4 *>(packed + termsf_off) + ps->term0;
    int4 *tdst = dst + NS;
    for (int k = threadIdx.x; k < nt; k += blockDim.x) tdst[k] = tsrc[k];
}

/* ------------------------------------------------------------------ K2: persistent FP32 evaluation */
template <int S, bool DEF, int MAXM, class Pol>
DEV void eval_f32_body(const JobTable &jt) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long s_item;
    __shared__ int s_job, s_abort;
    __shared__ double s_red[16][2 * (MAXM + 1)];
    __shared__ uint32_t s_fail[16];
    const PackedSector &sec = *reinterpret_cast<const PackedSector *>(smem);
    const PackedTermF *T = reinterpret_cast<const PackedTermF *>(smem + sizeof(PackedSector));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    int cur = -1, cur_job = -1;
    for (;;) {
        if (threadIdx.x == 0) {
            const long long it = (long long)atomicAdd(jt.counter, 1ull);
            s_item = it;
            s_job = it < jt.total_items ? find_job(jt, it) : 0;
            s_abort = it < jt.total_items ? job_aborted(jt.jobs[s_job]) : 0;
        }
        __syncthreads();
        const long long item = s_item;
        if (item >= jt.total_items) break;
        const int jb = s_job;
        const Job &J = jt.jobs[jb];
        const long long local = item - J.item_begin;
        if (s_abort) { /* the pass was stopped: its remaining items contribute nothing */
            if ((int)threadIdx.x < J.n_slots * 2) J.partials[local * J.n_slots * 2 + threadIdx.x] = 0.0;
            if (threadIdx.x == 0) J.part_fails[local] = 0;
            __syncthreads();
            continue;
        }
        const long long per_sector = (long long)J.m * J.chunks;
        const int ls = (int)(local / per_sector);
        const long long rem = local - (long long)ls * per_sector;
        const int shift = (int)(rem / J.chunks);
        const long long chunk = rem - (long long)shift * J.chunks;
        const int psec = J.sector_begin + ls;
        int level = -1; /* island level: the FP64 kernel has evaluated the island points and written the partial */
        if (J.sector_prec) {
            /* mixed pass: items of sectors evaluated in FP64 belong to the other kernel */
            const PackedSector *gps = reinterpret_cast<const PackedSector *>(J.packed + J.sectors_off) + psec;
            const int code = J.sector_prec[gps->orig_index];
            level = island_level(code);
            if (code != 1 && level < 0) {
                __syncthreads();
                continue;
            }
        }
        if (psec != cur || jb != cur_job) {
            stage_sector_f(J.packed, J.sectors_off, J.termsf_off, psec, smem);
            __syncthreads();
            cur = psec;
            cur_job = jb;
        }
        const Exps ex = Pol::exps(J);
        const Pol pol = Pol::make(T, sec, psec);
        const uint32_t n = J.n;
        const float invnf = 1.f / (float)n;
        const float lam = (float)J.lambda[sec.orig_index];
        uint32_t rj[S], aj[S], zs[S];
        float bj[S];
        const long long i0 = chunk * (long long)blockDim.x * jt.P + threadIdx.x;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            split_shift(J.shifts[6 * shift + j], n, aj[j], bj[j]);
            rj[j] = (uint32_t)(((unsigned long long)i0 * J.z[j]) % n);
            zs[j] = J.zstep[j];
        }
        float acc[2 * (MAXM + 1)], cmp[2 * (MAXM + 1)];
#pragma unroll
        for (int q = 0; q < 2 * (MAXM + 1); ++q) acc[q] = cmp[q] = 0.f;
        uint32_t fails = 0;
        const float rn = island_rn(n), xi = island_xi(level < 0 ? 0 : level);
        for (int p = 0; p < jt.P; ++p) {
            const long long i = i0 + (long long)p * blockDim.x;
            bool take = i < (long long)n;
            if (take && level >= 0) {
                uint32_t k[S];
#pragma unroll
                for (int j = 0; j < S; ++j) k[j] = shifted_index(rj[j], aj[j], n);
                take = !(island_key<S>(k, (unsigned)sec.sing_mask, rn) < xi);
            }
            if (take) {
                float x[S], y[S];
#pragma unroll
                for (int j = 0; j < S; ++j) lattice_f32(rj[j], aj[j], bj[j], n, invnf, x[j], y[j]);
                cf val[MAXM + 1];
                point_integrand_f<S, DEF, MAXM>(sec, pol, x, y, jt.r, lam, ex, val, fails);
#pragma unroll
                for (int m = 0; m <= MAXM; ++m) {
                    two_sum_acc(acc[2 * m], cmp[2 * m], val[m].x);
                    two_sum_acc(acc[2 * m + 1], cmp[2 * m + 1], val[m].y);
                }
            }
#pragma unroll
            for (int j = 0; j < S; ++j) {
                const uint32_t v = rj[j] + zs[j];
                rj[j] = v >= n ? v - n : v;
            }
        }
        /* warp: double-float shuffle tree; warps and items in FP64 */
#pragma unroll
        for (int q = 0; q < 2 * (MAXM + 1); ++q) {
            float s1 = acc[q], c1 = cmp[q];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const float so = __shfl_down_sync(0xffffffffu, s1, off);
                const float co = __shfl_down_sync(0xffffffffu, c1, off);
                two_sum_acc(s1, c1, so);
                c1 += co;
            }
            if (lane == 0) s_red[warp][q] = (double)s1 + (double)c1;
        }
        uint32_t f = fails;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) f += __shfl_down_sync(0xffffffffu, f, off);
        if (lane == 0) s_fail[warp] = f;
        __syncthreads();
        if (threadIdx.x < 32) {
            const int q = threadIdx.x;
            if (q < J.n_slots * 2) {
                double s2 = 0.0, c2 = 0.0;
                if (q < 2 * (MAXM + 1))
                    for (int w = 0; w < nwarps; ++w) kahan_add(s2, c2, s_red[w][q]);
                double *dst = &J.partials[local * J.n_slots * 2 + q];
                *dst = level >= 0 ? *dst + (s2 - c2) : s2 - c2;
            }
            if (q == 0) {
                uint32_t tf = 0;
                for (int w = 0; w < nwarps; ++w) tf += s_fail[w];
                J.part_fails[local] = level >= 0 ? J.part_fails[local] + tf : tf;
            }
        }
        __syncthreads();
    }
}

template <int S, bool DEF, int MAXM>
__global__ void __launch_bounds__(256) qmc_eval_kernel_f32(const __grid_constant__ JobTable jt) {
    eval_f32_body<S, DEF, MAXM, TabPolF<S>>(jt);
}

/* ================================================================== FP32 path, two lattice points per thread
 * The generated evaluators of the mixed pass evaluate two lattice points per thread, one in each lane of GB300's
 * packed FP32 instructions (__ffma2_rn, __fmul2_rn, __fadd2_rn): every arithmetic step of the per-point code is
 * issued once for both points, the staged coefficients are read once for both, and the control flow of the
 * subtraction subsets is shared.  Each lane rounds exactly as the scalar code of the one-point path does, so a
 * lane's value equals that path's value for its point.  Steps without a packed form run per lane with the scalar
 * code: the transcendentals and the reciprocals.
 * Coefficients are staged as (hi, hi, lo, lo): one 128-bit shared load gives both packed operands of a term. */
DEV float2 bc2(float v) { return make_float2(v, v); }
DEV float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
DEV float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
DEV float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
DEV float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
DEV float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
DEV float lane(float2 v, int k) { return k ? v.y : v.x; }

/* two complex numbers: lane a = (re.x, im.x), lane b = (re.y, im.y) */
struct c2 {
    float2 re, im;
};
DEV c2 mkc2(float2 re, float2 im) { return c2{re, im}; }
DEV c2 zero_c2() { return c2{bc2(0.f), bc2(0.f)}; }
DEV c2 cadd2(c2 a, c2 b) { return c2{add2(a.re, b.re), add2(a.im, b.im)}; }
DEV c2 cscale2(c2 a, float2 s) { return c2{mul2(a.re, s), mul2(a.im, s)}; }
/* as cmulf per lane: (fma(a.re, b.re, rn(-a.im b.im)), fma(a.re, b.im, rn(a.im b.re))) */
DEV c2 cmul2(c2 a, c2 b) { return c2{fma2(a.re, b.re, neg2(mul2(a.im, b.im))), fma2(a.re, b.im, mul2(a.im, b.re))}; }
/* a + (hi + lo) m for a staged coefficient (hi, hi, lo, lo), as cfma2f per lane */
DEV c2 cfma2c(const float4 &c, c2 m, c2 a) {
    const float2 h = make_float2(c.x, c.y), l = make_float2(c.z, c.w);
    return c2{fma2(h, m.re, fma2(l, m.re, a.re)), fma2(h, m.im, fma2(l, m.im, a.im))};
}
/* a + hi m, real (coefficients that only shape the contour deformation) */
DEV float2 rfma2h(const float4 &c, float2 m, float2 a) { return fma2(make_float2(c.x, c.y), m, a); }
/* a + (hi + lo) m, real */
DEV float2 rfma2c(const float4 &c, float2 m, float2 a) {
    return fma2(make_float2(c.x, c.y), m, fma2(make_float2(c.z, c.w), m, a));
}
DEV c2 cinv2(c2 a) {
    const float2 d2 = fma2(a.re, a.re, mul2(a.im, a.im));
    const float2 d = make_float2(__fdividef(1.f, d2.x), __fdividef(1.f, d2.y));
    return c2{mul2(a.re, d), neg2(mul2(a.im, d))};
}
/* the periodising transform of both points (transform_f per lane) */
DEV void transform2(int r, float2 x, float2 y, float2 &t, float2 &tm, float2 &w) {
    const bool la = x.x <= y.x, lb = x.y <= y.y;
    const float2 u = make_float2(la ? x.x : y.x, lb ? x.y : y.y);
    float2 p;
    switch (r) {
        case 0: p = u; break;
        case 1: p = mul2(mul2(u, u), fma2(bc2(-2.f), u, bc2(3.f))); break;
        case 2: p = mul2(mul2(mul2(u, u), u), fma2(u, fma2(bc2(6.f), u, bc2(-15.f)), bc2(10.f))); break;
        default: {
            const float2 u2 = mul2(u, u);
            p = mul2(mul2(u2, u2), fma2(u, fma2(u, fma2(bc2(-20.f), u, bc2(70.f)), bc2(-84.f)), bc2(35.f)));
        }
    }
    const float2 q = sub2(bc2(1.f), p);
    t = make_float2(la ? p.x : q.x, lb ? p.y : q.y);
    tm = make_float2(la ? q.x : p.x, lb ? q.y : p.y);
    const float2 xy = mul2(x, y);
    switch (r) {
        case 0: w = bc2(1.f); break;
        case 1: w = mul2(bc2(6.f), xy); break;
        case 2: w = mul2(mul2(bc2(30.f), xy), xy); break;
        default: w = mul2(mul2(mul2(bc2(140.f), xy), xy), xy); break;
    }
}

/* What the two-point kernels read of the staged sector's exponents at every point (stage_sector_f2 fills it): B_j and
   1/B_j as floats, and bit sets over the variables, tested where the exponents themselves would be loaded, compared and
   looped over. */
struct SectorConstF {
    float B[8], rB[8];
    unsigned a1, a2, more; /* A_j >= 1; A_j >= 2; A_j >= 3 */
    unsigned a, b, l;      /* A_j != 0; B_j != 0; B_j != 0 and A_j != -1 */
    float one;             /* 1 (see det_sym_f2) */
};
static __shared__ SectorConstF qmc_secf;

/* v^e, e known at compile time in the generated kernels */
DEV float2 rpow2(float2 v, int e) {
    float2 r = v;
    for (int i = e < 0 ? -e : e; i > 1; --i) r = mul2(r, v);
    return e < 0 ? make_float2(__frcp_rn(r.x), __frcp_rn(r.y)) : r;
}
DEV c2 cpow2(c2 z, int e) {
    c2 r = z;
    for (int i = e < 0 ? -e : e; i > 1; --i) r = cmul2(r, z);
    return e < 0 ? cinv2(r) : r;
}
/* v prod_j tt_j^{A_j} over A_j > 0 */
template <int S>
DEV float2 mono2(const PackedSector &s, float2 v, const float2 *tt) {
#pragma unroll
    for (int j = 0; j < S; ++j) {
        if ((qmc_secf.a1 >> j) & 1u) v = mul2(v, tt[j]);
        if ((qmc_secf.a2 >> j) & 1u) v = mul2(v, tt[j]);
        if ((qmc_secf.more >> j) & 1u)
            for (int k = 2; k < s.A[j]; ++k) v = mul2(v, tt[j]);
    }
    return v;
}

/* det(I - i lam A) at both lanes' points for S >= 4: det_sym_f per lane, in packed arithmetic over the lanes.  n: the
   imaginary parts -lam b_jk of the symmetric matrix (packed upper triangle), whose real part is the identity: the
   first elimination step works on imaginary numbers only and keeps 15 complex entries (S = 6) alive instead of 21.
   Bound by issue and the FP32 pipe: 330 packed instructions for both points; per lane it took 330 twice, and as many
   moves to swap real and imaginary parts.
   Signs are folded into the factors, so that each difference is one packed addition (negation is exact).  Where a product
   is rounded before it is added, the addition is an FMA with a factor 1 that the compiler does not know (it would fuse
   the packed product into a packed addition). */
template <int S>
DEV c2 det_sym_f2(const float2 (&n)[S * (S + 1) / 2]) {
    auto at = [](int i, int j) { return i * S - i * (i - 1) / 2 + (j - i); }; /* i <= j */
    const float2 one = bc2(1.f), rt1 = bc2(qmc_secf.one);
    auto add_rn = [&](float2 a, float2 b) { return fma2(a, rt1, b); };
    c2 N[S * (S + 1) / 2];
    {
        const float2 m2 = fma2(n[0], n[0], one);
        const float2 d = make_float2(__fdividef(1.f, m2.x), __fdividef(1.f, m2.y));
        const float2 iy = neg2(mul2(n[0], d)); /* 1 / (1 + i n_0) = d + i iy */
#pragma unroll
        for (int i = 1; i < S; ++i) {
            const float2 u = mul2(n[at(0, i)], iy), v = mul2(n[at(0, i)], d); /* row 0 over the pivot: -u + i v */
#pragma unroll
            for (int j = i; j < S; ++j) {
                const float2 p = mul2(v, n[at(0, j)]);
                N[at(i, j)] = c2{i == j ? add_rn(p, one) : p, add_rn(n[at(i, j)], mul2(u, n[at(0, j)]))};
            }
        }
    }
    /* (1 + i n_0) times the second pivot */
    c2 det = c2{add_rn(N[at(1, 1)].re, neg2(mul2(n[0], N[at(1, 1)].im))), add_rn(N[at(1, 1)].im, mul2(n[0], N[at(1, 1)].re))};
#pragma unroll
    for (int k = 1; k < S; ++k) {
        const c2 dk = N[at(k, k)];
        if (k > 1) det = cmul2(det, dk);
        if (k + 1 < S) {
            const c2 iv = cinv2(dk);
            const float2 mx = neg2(iv.re), my = neg2(iv.im);
#pragma unroll
            for (int i = k + 1; i < S; ++i) {
                const c2 a = N[at(k, i)];
                /* l = -a / d_k and m = -Im l */
                const c2 l = c2{fma2(a.re, mx, mul2(a.im, iv.im)), fma2(a.re, my, mul2(a.im, mx))};
                const float2 m = fma2(a.re, iv.im, mul2(a.im, iv.re));
#pragma unroll
                for (int j = i; j < S; ++j) {
                    const c2 w = N[at(k, j)];
                    N[at(i, j)].re = add_rn(N[at(i, j)].re, fma2(l.re, w.re, mul2(m, w.im)));
                    N[at(i, j)].im = add2(N[at(i, j)].im, fma2(l.re, w.im, mul2(l.im, w.re)));
                }
            }
        }
    }
    return det;
}

/* det_deform_f per lane for S <= 3, in packed arithmetic */
template <int S>
DEV c2 det_deform_f2(const float2 (&A)[S][S], float lam) {
    const float2 l = bc2(lam), ml = bc2(-lam);
    if constexpr (S == 1) {
        return c2{bc2(1.f), mul2(ml, A[0][0])};
    } else if constexpr (S == 2) {
        const float2 tr = add2(A[0][0], A[1][1]);
        const float2 dt = fma2(A[0][0], A[1][1], neg2(mul2(A[0][1], A[1][0])));
        return c2{fma2(mul2(ml, l), dt, bc2(1.f)), mul2(ml, tr)};
    } else {
        const float2 tr = add2(add2(A[0][0], A[1][1]), A[2][2]);
        const float2 p01 = fma2(A[0][0], A[1][1], neg2(mul2(A[0][1], A[1][0])));
        const float2 p02 = fma2(A[0][0], A[2][2], neg2(mul2(A[0][2], A[2][0])));
        const float2 p12 = fma2(A[1][1], A[2][2], neg2(mul2(A[1][2], A[2][1])));
        const float2 e2 = add2(add2(p01, p02), p12);
        const float2 q1 = fma2(A[1][0], A[2][2], neg2(mul2(A[1][2], A[2][0])));
        const float2 q2 = fma2(A[1][0], A[2][1], neg2(mul2(A[1][1], A[2][0])));
        const float2 dt = fma2(A[0][2], q2, fma2(A[0][0], p12, neg2(mul2(A[0][1], q1))));
        const float2 l2 = mul2(l, l);
        return c2{fma2(neg2(l2), e2, bc2(1.f)), fma2(mul2(l2, l), dt, mul2(ml, tr))};
    }
}

/* G at the points tt of both lanes (eval_G_f per lane): its eps^0 value G0 and, with needX, the eps-coefficient X of
   its logarithm.  First the undeformed class, where everything is real. */
template <int S, class Pol>
DEV void eval_G_f2(const PackedSector &s, const Pol &P, unsigned Y, const float2 *tt, const float2 *Lt, bool needX,
                   const Exps &ex, float2 &G0, float2 &X) {
    float2 U, F;
    P.UFr(Y, tt, U, F);
    if (s.kind == 1) F = neg2(F);
    float2 g = bc2(s.Df);
    if (ex.eU0 != 0) g = mul2(g, rpow2(U, ex.eU0));
    if (ex.eF0 != 0) g = mul2(g, rpow2(F, -ex.eF0));
    G0 = mono2<S>(s, g, tt);
    X = bc2(0.f);
    if (needX) {
        float2 a = ex.eU1 != 0 ? rpow2(U, ex.eU1) : bc2(1.f);
        if (ex.eF1 != 0) a = mul2(a, rpow2(F, -ex.eF1));
        X = make_float2(__logf(a.x), __logf(a.y));
#pragma unroll
        for (int j = 0; j < S; ++j)
            if ((qmc_secf.l >> j) & 1u) X = fma2(bc2(qmc_secf.B[j]), Lt[j], X);
    }
}

/* Deformed sectors, first half: the contour of Eq. 14 at the points tt of both lanes, z_j = t_j (1 - i d_j) with
   d_j = lam (1 - t_j) dF/dt_j, and its Jacobian. */
template <int S, class Pol>
DEV void deform_f2(const Pol &P, unsigned Y, const float2 *tt, const float2 *ttm, float lam, float2 *g, c2 &detJ) {
    {
        float2 h[S * (S + 1) / 2];
        P.GH(Y, tt, g, h);
        if constexpr (S >= 4) {
            float2 sq[S];
#pragma unroll
            for (int j = 0; j < S; ++j) {
                const float2 pj = mul2(tt[j], ttm[j]);
                sq[j] = make_float2(pj.x > 0.f ? pj.x * rsqrtf(pj.x) : 0.f, pj.y > 0.f ? pj.y * rsqrtf(pj.y) : 0.f);
            }
            const float2 ml = bc2(-lam);
            int p = 0;
#pragma unroll
            for (int j = 0; j < S; ++j) {
#pragma unroll
                for (int i = j; i < S; ++i) {
                    h[p] = mul2(ml, (i == j) ? fma2(sub2(ttm[j], tt[j]), g[j], mul2(mul2(tt[j], ttm[j]), h[p]))
                                                : mul2(mul2(sq[j], sq[i]), h[p]));
                    ++p;
                }
            }
            detJ = det_sym_f2<S>(h);
        } else {
            float2 A[S][S];
            int p = 0;
#pragma unroll
            for (int j = 0; j < S; ++j) {
#pragma unroll
                for (int i = j; i < S; ++i) {
                    A[j][i] = mul2(mul2(tt[j], ttm[j]), h[p]);
                    if (i != j) A[i][j] = mul2(mul2(tt[i], ttm[i]), h[p]);
                    ++p;
                }
            }
#pragma unroll
            for (int j = 0; j < S; ++j) A[j][j] = fma2(sub2(ttm[j], tt[j]), g[j], A[j][j]);
            detJ = det_deform_f2<S>(A, lam);
        }
    }
#pragma unroll
    for (int j = 0; j < S; ++j) g[j] = mul2(mul2(bc2(lam), ttm[j]), g[j]);
}

/* Second half: G at the deformed points.  live: lanes whose point is evaluated (a sign failure is counted only there). */
template <int S, class Pol>
DEV void value_f2(const PackedSector &s, const Pol &P, unsigned Y, const float2 *tt, const float2 *g, c2 detJ, bool needX,
                  const Exps &ex, const bool (&live)[2], c2 &G0, c2 &X, uint32_t &fails) {
    c2 z[S];
#pragma unroll
    for (int j = 0; j < S; ++j) z[j] = c2{tt[j], neg2(mul2(tt[j], g[j]))};
    c2 U, F;
    P.UFc(Y, z, ex.eU0 != 0 || needX, U, F);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float fr = lane(F.re, k), fi = lane(F.im, k);
        fails += (live[k] && fi > QMC_F32_SIGN_NOISE * (fabsf(fr) + fabsf(fi))) ? 1u : 0u;
    }
    c2 G = cscale2(detJ, bc2(s.Df));
    if (ex.eU0 != 0) G = cmul2(G, cpow2(U, ex.eU0));
    if (ex.eF0 != 0) G = cmul2(G, cpow2(F, -ex.eF0));
    if (qmc_secf.a) {
        if (qmc_secf.a1) G = cscale2(G, mono2<S>(s, bc2(1.f), tt));
#pragma unroll
        for (int j = 0; j < S; ++j)
            if ((qmc_secf.a >> j) & 1u) G = cmul2(G, cpow2(c2{bc2(1.f), neg2(g[j])}, s.A[j]));
    }
    G0 = G;
    X = zero_c2();
    if (needX) {
        const float2 eU1 = bc2((float)ex.eU1), eF1 = bc2((float)ex.eF1);
        const float2 U2 = fma2(U.re, U.re, mul2(U.im, U.im)), F2 = fma2(F.re, F.re, mul2(F.im, F.im));
        const float2 lU = make_float2(0.5f * __logf(U2.x), 0.5f * __logf(U2.y));
        const float2 lF = make_float2(0.5f * __logf(F2.x), 0.5f * __logf(F2.y));
        const float2 aU = make_float2(atan2f(U.im.x, U.re.x), atan2f(U.im.y, U.re.y));
        const float2 aF = make_float2(arg_mi0f(F.re.x, F.im.x), arg_mi0f(F.re.y, F.im.y));
        float2 xr = sub2(mul2(lU, eU1), mul2(lF, eF1)), xi = sub2(mul2(aU, eU1), mul2(aF, eF1));
        /* log q_j with q_j = 1 - i d_j: (log(1 + d_j^2) / 2, -atan d_j) */
        float2 lr = bc2(0.f);
#pragma unroll
        for (int j = 0; j < S; ++j) {
            if ((qmc_secf.b >> j) & 1u) {
                const float2 Bj = bc2(qmc_secf.B[j]), d = g[j];
                if ((qmc_secf.l >> j) & 1u) xr = fma2(Bj, make_float2(__logf(tt[j].x), __logf(tt[j].y)), xr);
                const float2 q2 = fma2(d, d, bc2(1.f));
                lr = fma2(Bj, make_float2(__logf(q2.x), __logf(q2.y)), lr);
                xi = fma2(neg2(Bj), make_float2(atanf(d.x), atanf(d.y)), xi);
            }
        }
        X = c2{fma2(bc2(0.5f), lr, xr), xi};
    }
}

/* Series values of the two classes: real pairs and complex pairs */
DEV float2 vzero2(float2) { return bc2(0.f); }
DEV c2 vzero2(c2) { return zero_c2(); }
DEV float2 vmadd2(float2 o, float2 g, float2 V) { return add2(o, mul2(g, V)); }
DEV c2 vmadd2(c2 o, c2 g, float2 V) { return cadd2(o, cscale2(g, V)); }
DEV float2 vnext2(float2 g, float2 X) { return mul2(g, X); }
DEV c2 vnext2(c2 g, c2 X) { return cmul2(g, X); }
DEV float2 vscale2(float2 g, float f) { return mul2(g, bc2(f)); }
DEV c2 vscale2(c2 g, float f) { return cscale2(g, bc2(f)); }
DEV c2 to_c2(float2 v) { return c2{v, bc2(0.f)}; }
DEV c2 to_c2(c2 v) { return v; }

/* V times the factor of a singular variable (subset_factor of the FP64 path), for series up to eps^M; a: the variable's
   series, with 1/B in the place of eps^0 */
template <int M, int N>
DEV void subset_factor2(float2 (&V)[N], const float2 *a, bool inY) {
    float2 f[M + 1];
    f[0] = inY ? a[0] : bc2(0.f);
#pragma unroll
    for (int n = 1; n <= M; ++n) f[n] = inY ? neg2(a[n]) : a[n];
#pragma unroll
    for (int n = M; n >= 0; --n) {
        float2 acc = bc2(0.f);
#pragma unroll
        for (int k = 0; k <= n; ++k) acc = fma2(V[k], f[n - k], acc);
        V[n] = acc;
    }
}

/* o += G_Y(eps) V_Y(eps) for the subset with the bits `count`, series up to eps^M: V_Y from the shared product `pre` of
   the first np variables and the factors of the others */
template <int M, int N, class V2>
DEV void subset_add2(V2 (&o)[N], V2 g, V2 X, const float2 (&pre)[N], int np, int sigma, unsigned count,
                     const float2 (*a)[N], int need) {
    float2 V[N];
#pragma unroll
    for (int n = 0; n <= M; ++n) V[n] = pre[n];
    for (int i = np; i < sigma; ++i) subset_factor2<M>(V, a[i], (count >> i) & 1u);
#pragma unroll
    for (int n = 0; n <= M; ++n) {
        if (n > need) break;
#pragma unroll
        for (int k = 0; k + n <= M; ++k) o[n + k] = vmadd2(o[n + k], g, V[k]);
        if (n < M) {
            g = vnext2(g, X);
            if (n > 0) g = vscale2(g, 1.f / (n + 1));
        }
    }
}

template <int MAXM, class V2>
DEV void subset_add2(int M, V2 (&o)[MAXM + 1], V2 g, V2 X, const float2 (&pre)[MAXM + 1], int np, int sigma, unsigned count,
                     const float2 (*a)[MAXM + 1], int need) {
    switch (MAXM == 0 ? 0 : M) {
        case 0: subset_add2<0>(o, g, X, pre, np, sigma, count, a, need); break;
        case 1: if constexpr (MAXM >= 1) subset_add2<1>(o, g, X, pre, np, sigma, count, a, need); break;
        case 2: if constexpr (MAXM >= 2) subset_add2<2>(o, g, X, pre, np, sigma, count, a, need); break;
        case 3: if constexpr (MAXM >= 3) subset_add2<3>(o, g, X, pre, np, sigma, count, a, need); break;
        case 4: if constexpr (MAXM >= 4) subset_add2<4>(o, g, X, pre, np, sigma, count, a, need); break;
        default: break;
    }
}

/* The transform of both lanes' points (x, y = 1 - x); live[k]: lane k holds a lattice point, and on return whether its
   weight is positive.  A lane without a point takes the other lane's (its value is discarded).  false: neither lane. */
template <int S>
DEV bool pair_setup(const float2 *x, const float2 *y, int r, bool (&live)[2], float2 (&t)[S], float2 (&tm)[S], float2 &w) {
#pragma unroll
    for (int j = 0; j < S; ++j) {
        float2 wj;
        transform2(r, x[j], y[j], t[j], tm[j], wj);
        w = j == 0 ? wj : mul2(w, wj);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        bool bad = !(lane(w, k) > 0.f);
#pragma unroll
        for (int j = 0; j < S; ++j) bad |= !(lane(t[j], k) > 0.f) || !(lane(tm[j], k) > 0.f);
        live[k] = live[k] && !bad;
    }
    if (!live[0] && !live[1]) return false;
    if (!live[0] || !live[1]) {
        const int from = live[0] ? 0 : 1;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            t[j] = bc2(lane(t[j], from));
            tm[j] = bc2(lane(tm[j], from));
        }
        w = bc2(lane(w, from));
    }
    return true;
}

/* logarithms of the variables that need one, and the series eps t^{-1 + B eps} of the singular ones */
template <int S, int MAXM>
DEV void pair_series(const PackedSector &s, const float2 (&t)[S], float2 (&Lt)[S], float2 (&a)[S][MAXM + 1]) {
    const int M = s.M;
    int i = 0;
#pragma unroll
    for (int j = 0; j < S; ++j) {
        const bool sing = ((unsigned)s.sing_mask >> j) & 1u;
        Lt[j] = bc2(0.f);
        if (MAXM > 0 && M > 0 && (sing || ((qmc_secf.l >> j) & 1u))) Lt[j] = make_float2(__logf(t[j].x), __logf(t[j].y));
        if (!sing) continue;
        a[i][0] = bc2(qmc_secf.rB[j]); /* the place of eps^0 holds 1/B_j */
        if (MAXM > 0 && M > 0) {
            float2 c = make_float2(__fdividef(1.f, t[j].x), __fdividef(1.f, t[j].y));
            const float2 bl = mul2(bc2(qmc_secf.B[j]), Lt[j]);
#pragma unroll
            for (int n = 1; n <= MAXM; ++n) {
                a[i][n] = c;
                if (n >= M) break;
                c = mul2(c, n == 1 ? bl : make_float2(bl.x / n, bl.y / n));
            }
        }
        ++i;
    }
}

/* w(x) * (sector integrand) at the points (x, y = 1 - x) of both lanes, as point_integrand_f per lane; live[k]:
   lane k holds a lattice point (its value is zero otherwise).
   As in the FP64 path, the series of the singular variables and the products of all but the last of them are made once
   per pair of points (local memory), and G_Y is taken only to the order at which its subset contributes: what is left
   out are sums and products with exact zeros, and logarithms that nothing uses.  Bound by instruction issue; with the
   same point values, mixed passes (16 shifts): massive box n = 1048573 1.05 -> 0.86 ms, four-pole double box n = 65521
   (all FP32) 12.4 -> 9.1 ms. */
template <int S, bool DEF, int MAXM, class Pol>
DEV void point_integrand_f2(const PackedSector &s, const Pol &P, const float2 *x, const float2 *y, int r, float lam,
                            const Exps &ex, bool (&live)[2], c2 (&out)[MAXM + 1], uint32_t &fails) {
    typedef typename Select<DEF, c2, float2>::type V2;
    float2 t[S], tm[S], w;
#pragma unroll
    for (int n = 0; n <= MAXM; ++n) out[n] = zero_c2();
    if (!pair_setup<S>(x, y, r, live, t, tm, w)) return;
    const int M = s.M, sigma = s.sigma;
    const unsigned smask = (unsigned)s.sing_mask;
    float2 Lt[S], a[S][MAXM + 1];
    pair_series<S, MAXM>(s, t, Lt, a);
    constexpr int NPRE = S < 4 ? S : 4;
    float2 pre[1 << (NPRE - 1)][MAXM + 1];
    const int np = sigma < NPRE ? (sigma > 0 ? sigma - 1 : 0) : NPRE - 1;
#pragma unroll
    for (int n = 0; n <= MAXM; ++n) pre[0][n] = bc2(n == 0 ? 1.f : 0.f);
    for (int i = 0; i < np; ++i)
        for (int k = 0; k < (1 << i); ++k) {
            float2 V[MAXM + 1], W[MAXM + 1];
#pragma unroll
            for (int n = 0; n <= MAXM; ++n) V[n] = W[n] = pre[k][n];
            subset_factor2<MAXM>(V, a[i], false);
            subset_factor2<MAXM>(W, a[i], true);
#pragma unroll
            for (int n = 0; n <= MAXM; ++n) {
                pre[k][n] = V[n];
                pre[k + (1 << i)][n] = W[n];
            }
        }
    V2 o[MAXM + 1];
#pragma unroll
    for (int n = 0; n <= MAXM; ++n) o[n] = vzero2(o[n]);
    unsigned Y = 0, count = 0;
    do {
        float2 tt[S], ttm[S];
#pragma unroll
        for (int j = 0; j < S; ++j) {
            const bool zj = (Y >> j) & 1u;
            tt[j] = zj ? bc2(0.f) : t[j];
            ttm[j] = zj ? bc2(1.f) : tm[j];
        }
        const int need = M - sigma + __popc(count); /* highest order of eps to which G_Y is needed */
        V2 G0, X;
        if constexpr (DEF) {
            float2 d[S];
            c2 detJ;
            deform_f2<S>(P, Y, tt, ttm, lam, d, detJ);
            value_f2<S>(s, P, Y, tt, d, detJ, MAXM > 0 && need > 0, ex, live, G0, X, fails);
        } else
            eval_G_f2<S>(s, P, Y, tt, Lt, MAXM > 0 && need > 0, ex, G0, X);
        const unsigned low = count & ((1u << np) - 1u);
        subset_add2<MAXM>(M, o, G0, X, pre[low], np, sigma, count, a, need);
        ++count;
        Y = (Y - smask) & smask;
    } while (Y != 0);
#pragma unroll
    for (int n = 0; n <= MAXM; ++n) {
        out[n] = cscale2(to_c2(o[n]), w);
        if (!live[0]) out[n] = c2{make_float2(0.f, out[n].re.y), make_float2(0.f, out[n].im.y)};
        if (!live[1]) out[n] = c2{make_float2(out[n].re.x, 0.f), make_float2(out[n].im.x, 0.f)};
    }
}

/* stage a sector for the two-point path: the record, then each term's coefficient as (hi, hi, lo, lo) */
DEV void stage_sector_f2(const unsigned char *packed, int64_t sectors_off, int64_t termsf_off, int psec,
                         unsigned char *smem) {
    const PackedSector *ps = reinterpret_cast<const PackedSector *>(packed + sectors_off) + psec;
    const int4 *src = reinterpret_cast<const int4 *>(ps);
    int4 *dst = reinterpret_cast<int4 *>(smem);
    constexpr int NS = (int)(sizeof(PackedSector) / 16);
    for (int k = threadIdx.x; k < NS; k += blockDim.x) dst[k] = src[k];
    if (threadIdx.x < 8) {
        const float B = (float)ps->B[threadIdx.x];
        qmc_secf.B[threadIdx.x] = B;
        qmc_secf.rB[threadIdx.x] = __fdividef(1.f, B); /* used for singular variables only: B != 0 there */
        const int A = ps->A[threadIdx.x];
        const unsigned m = 0xffu;
        const unsigned a1 = __ballot_sync(m, A >= 1), a2 = __ballot_sync(m, A >= 2), more = __ballot_sync(m, A >= 3);
        const unsigned an = __ballot_sync(m, A != 0), b = __ballot_sync(m, B != 0.f), l = __ballot_sync(m, B != 0.f && A != -1);
        if (threadIdx.x == 0) {
            qmc_secf.a1 = a1;
            qmc_secf.a2 = a2;
            qmc_secf.more = more;
            qmc_secf.a = an;
            qmc_secf.b = b;
            qmc_secf.l = l;
            qmc_secf.one = 1.f;
        }
    }
    const int nt = ps->n_terms;
    const PackedTermF *tsrc = reinterpret_cast<const PackedTermF *>(packed + termsf_off) + ps->term0;
    float4 *tdst = reinterpret_cast<float4 *>(dst + NS);
    for (int k = threadIdx.x; k < nt; k += blockDim.x) {
        const float hi = tsrc[k].hi, lo = tsrc[k].lo;
        tdst[k] = make_float4(hi, hi, lo, lo);
    }
}

/* Points p and p + 1 of the thread whose first lattice index is i0 (stride: threads of the item): coordinates x and 1 - x
   of both lanes, and which of them are evaluated here; steps the residues r_j past both. */
template <int S>
DEV void next_pair(long long i0, int p, int P, int stride, uint32_t n, float invnf, int level, unsigned smask, float rn, float xi,
                   uint32_t (&rj)[S], const uint32_t (&aj)[S], const float (&bj)[S], const uint32_t (&zs)[S], bool (&live)[2],
                   float2 (&x)[S], float2 (&y)[S]) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const long long i = i0 + (long long)(p + k) * stride;
        live[k] = (p + k < P) && i < (long long)n;
        if (live[k] && level >= 0) {
            uint32_t kk[S];
#pragma unroll
            for (int j = 0; j < S; ++j) kk[j] = shifted_index(rj[j], aj[j], n);
            live[k] = !(island_key<S>(kk, smask, rn) < xi);
        }
#pragma unroll
        for (int j = 0; j < S; ++j) {
            float xv, yv;
            lattice_f32(rj[j], aj[j], bj[j], n, invnf, xv, yv);
            if (k == 0) {
                x[j].x = xv;
                y[j].x = yv;
            } else {
                x[j].y = xv;
                y[j].y = yv;
            }
            const uint32_t v = rj[j] + zs[j];
            rj[j] = v >= n ? v - n : v;
        }
    }
}

/* adds both lanes' values to a thread's sums, lane a first */
template <int MAXM>
DEV void add_pair(float (&acc)[2 * (MAXM + 1)], float (&cmp)[2 * (MAXM + 1)], const c2 (&val)[MAXM + 1], const bool (&live)[2]) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (!live[k]) continue;
#pragma unroll
        for (int m = 0; m <= MAXM; ++m) {
            two_sum_acc(acc[2 * m], cmp[2 * m], lane(val[m].re, k));
            two_sum_acc(acc[2 * m + 1], cmp[2 * m + 1], lane(val[m].im, k));
        }
    }
}

/* a warp's sums: double-float shuffle tree; s_red, s_fail: the warp's place */
template <int MAXM>
DEV void warp_sums(const float (&acc)[2 * (MAXM + 1)], const float (&cmp)[2 * (MAXM + 1)], uint32_t fails, double *s_red,
                   uint32_t *s_fail) {
    const int lane_id = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < 2 * (MAXM + 1); ++q) {
        float s1 = acc[q], c1 = cmp[q];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const float so = __shfl_down_sync(0xffffffffu, s1, off);
            const float co = __shfl_down_sync(0xffffffffu, c1, off);
            two_sum_acc(s1, c1, so);
            c1 += co;
        }
        if (lane_id == 0) s_red[q] = (double)s1 + (double)c1;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) fails += __shfl_down_sync(0xffffffffu, fails, off);
    if (lane_id == 0) *s_fail = fails;
}

/* an item's partial from its warps' sums (compensated, in order), written by the item's first 32 threads (q: thread);
   add: to what the FP64 kernel left there for the island points */
template <int MAXM>
DEV void write_partial(const Job &J, long long local, int q, const double (*s_red)[2 * (MAXM + 1)], const uint32_t *s_fail,
                       int nwarps, bool add) {
    if (q < J.n_slots * 2) {
        double s2 = 0.0, c2v = 0.0;
        if (q < 2 * (MAXM + 1))
            for (int w = 0; w < nwarps; ++w) kahan_add(s2, c2v, s_red[w][q]);
        double *dst = &J.partials[local * J.n_slots * 2 + q];
        *dst = add ? *dst + (s2 - c2v) : s2 - c2v;
    }
    if (q == 0) {
        uint32_t tf = 0;
        for (int w = 0; w < nwarps; ++w) tf += s_fail[w];
        J.part_fails[local] = add ? J.part_fails[local] + tf : tf;
    }
}

/* ------------------------------------------------------------------ K2x2: persistent FP32 evaluation, two points
   per thread (generated evaluators).  Work items and their partials are those of eval_f32_body; a thread takes its
   P points in pairs (p, p + 1) and accumulates lane a before lane b, i.e. in the one-point path's order. */
template <int S, bool DEF, int MAXM, class Pol>
DEV void eval_f32x2_body(const JobTable &jt) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long s_item;
    __shared__ int s_job, s_abort;
    __shared__ double s_red[16][2 * (MAXM + 1)];
    __shared__ uint32_t s_fail[16];
    const PackedSector &sec = *reinterpret_cast<const PackedSector *>(smem);
    const float4 *T = reinterpret_cast<const float4 *>(smem + sizeof(PackedSector));
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    int cur = -1, cur_job = -1;
    for (;;) {
        if (threadIdx.x == 0) {
            const long long it = (long long)atomicAdd(jt.counter, 1ull);
            s_item = it;
            s_job = it < jt.total_items ? find_job(jt, it) : 0;
            s_abort = it < jt.total_items ? job_aborted(jt.jobs[s_job]) : 0;
        }
        __syncthreads();
        const long long item = s_item;
        if (item >= jt.total_items) break;
        const int jb = s_job;
        const Job &J = jt.jobs[jb];
        const long long local = item - J.item_begin;
        if (s_abort) { /* the pass was stopped: its remaining items contribute nothing */
            if ((int)threadIdx.x < J.n_slots * 2) J.partials[local * J.n_slots * 2 + threadIdx.x] = 0.0;
            if (threadIdx.x == 0) J.part_fails[local] = 0;
            __syncthreads();
            continue;
        }
        const long long per_sector = (long long)J.m * J.chunks;
        const int ls = (int)(local / per_sector);
        const long long rem = local - (long long)ls * per_sector;
        const int shift = (int)(rem / J.chunks);
        const long long chunk = rem - (long long)shift * J.chunks;
        const int psec = J.sector_begin + ls;
        int level = -1; /* island level: the FP64 kernel has evaluated the island points and written the partial */
        if (J.sector_prec) {
            const PackedSector *gps = reinterpret_cast<const PackedSector *>(J.packed + J.sectors_off) + psec;
            const int code = J.sector_prec[gps->orig_index];
            level = island_level(code);
            if (code != 1 && level < 0) {
                __syncthreads();
                continue;
            }
        }
        if (psec != cur || jb != cur_job) {
            stage_sector_f2(J.packed, J.sectors_off, J.termsf_off, psec, smem);
            __syncthreads();
            cur = psec;
            cur_job = jb;
        }
        const Exps ex = Pol::exps(J);
        const Pol pol = Pol::make(T, sec, psec);
        const uint32_t n = J.n;
        const float invnf = 1.f / (float)n;
        const float lam = (float)J.lambda[sec.orig_index];
        uint32_t rj[S], aj[S], zs[S];
        float bj[S];
        const long long i0 = chunk * (long long)blockDim.x * jt.P + threadIdx.x;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            split_shift(J.shifts[6 * shift + j], n, aj[j], bj[j]);
            rj[j] = (uint32_t)(((unsigned long long)i0 * J.z[j]) % n);
            zs[j] = J.zstep[j];
        }
        float acc[2 * (MAXM + 1)], cmp[2 * (MAXM + 1)];
#pragma unroll
        for (int q = 0; q < 2 * (MAXM + 1); ++q) acc[q] = cmp[q] = 0.f;
        uint32_t fails = 0;
        const float rn = island_rn(n), xi = island_xi(level < 0 ? 0 : level);
        for (int p = 0; p < jt.P; p += 2) {
            bool live[2];
            float2 x[S], y[S];
            next_pair<S>(i0, p, jt.P, blockDim.x, n, invnf, level, (unsigned)sec.sing_mask, rn, xi, rj, aj, bj, zs, live, x, y);
            if (live[0] || live[1]) {
                c2 val[MAXM + 1];
                point_integrand_f2<S, DEF, MAXM>(sec, pol, x, y, jt.r, lam, ex, live, val, fails);
                add_pair<MAXM>(acc, cmp, val, live);
            }
        }
        warp_sums<MAXM>(acc, cmp, fails, s_red[warp], &s_fail[warp]);
        __syncthreads();
        if (threadIdx.x < 32) write_partial<MAXM>(J, local, threadIdx.x, s_red, s_fail, nwarps, level >= 0);
        __syncthreads();
    }
}

/* ------------------------------------------------------------------ K2x2 in phases: deformed sectors of 5 and 6 dimensions
 * A pair of points of such a sector runs through 2400 instructions per zeroed subset, 38 KB of straight-line code of
 * which nothing repeats.  An SM partition issues one instruction per cycle from a 32 KB instruction cache, 0.4 per warp
 * from the next level and 0.17 from L2 (measured with loops of 2 KB to 256 KB): with three independent blocks per SM a
 * warp spent 2.5 of 6.8 cycles per instruction waiting for instructions, and more where the blocks were in different
 * sectors.  So all sixteen warps of an SM form one block that goes through the code in two phases per subset, each
 * short enough for that cache (contour and Jacobian; value and accumulation), over `pairs` pairs of points per thread,
 * with a barrier between them: a phase's code is fetched once for 4 warps x `pairs` passes.  What a pair carries from
 * phase to phase (coordinates, contour, Jacobian, series: 26 packed pairs for S = 6, MAXM = 2) lies in shared memory,
 * 208 bytes per pair and thread.  The block works on consecutive items of one sector, one per group of jt.block threads
 * (the threads of an item in the other kernels), so that items, their partials and their order of summation are those
 * of every other kernel.  item_begin and total_items count such sets of items here.
 * Measured (16 shifts), determinant per lane with three blocks per SM -> packed determinant and shorter series
 * with three blocks -> in phases: non-planar double box n = 3001 0.78, 0.71 -> 0.46 ms, n = 16381 2.1 -> 1.85 ms,
 * n = 1048573 115.7, 98-100 -> 103.0 ms; planar double box n = 50021 6.98, 5.92 -> 4.87 ms: three blocks stay 3 % ahead
 * only where every block is in the same sector for long.  What bounds it now is the FP32 pipe's operand ports: a packed
 * FMA with three distinct register pairs takes 3 cycles of a partition, a packed product 2; some 3000 cycles of 5200
 * per pair and subset.  384 threads, one pair in flight, or a barrier after the second phase: 0 to 9 % slower. */
template <int S, int MAXM>
struct PairState {
    enum { T = 0, TM = S, D = 2 * S, DET = 3 * S, O = 3 * S + 2, SIZE = 3 * S + 2 + 2 * (MAXM + 1) };
};

template <int S, int MAXM, class Pol>
DEV void eval_f32x2_phased_body(const JobTable &jt) {
    typedef PairState<S, MAXM> PS;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long s_item;
    __shared__ int s_job, s_abort;
    __shared__ double s_red[QMC_PHASED_THREADS / 32][2 * (MAXM + 1)];
    __shared__ uint32_t s_fail[QMC_PHASED_THREADS / 32];
    const PackedSector &sec = *reinterpret_cast<const PackedSector *>(smem);
    const float4 *T = reinterpret_cast<const float4 *>(smem + sizeof(PackedSector));
    float2 *state = reinterpret_cast<float2 *>(smem + jt.state_off) + threadIdx.x; /* [pair][value][thread] */
    const int stride = jt.block, groups = QMC_PHASED_THREADS / stride;
    const int group = threadIdx.x / stride, tl = threadIdx.x - group * stride;
    const int warp = threadIdx.x >> 5, nwarps = stride >> 5;
    auto st = [&](int q, int k) -> float2 & { return state[(q * PS::SIZE + k) * QMC_PHASED_THREADS]; };
    int cur = -1, cur_job = -1;
    for (;;) {
        if (threadIdx.x == 0) {
            const long long it = (long long)atomicAdd(jt.counter, 1ull);
            s_item = it;
            s_job = it < jt.total_items ? find_job(jt, it) : 0;
            s_abort = it < jt.total_items ? job_aborted(jt.jobs[s_job]) : 0;
        }
        __syncthreads();
        if (s_item >= jt.total_items) break;
        const int jb = s_job;
        const Job &J = jt.jobs[jb];
        const long long per_sector = (long long)J.m * J.chunks, sets = (per_sector + groups - 1) / groups;
        const long long set = s_item - J.item_begin;
        const int ls = (int)(set / sets);
        const long long rem = (set - (long long)ls * sets) * groups + group; /* this group's item within the sector */
        const bool have = group < groups && rem < per_sector; /* groups x jt.block threads may be fewer than the block */
        const long long local = (long long)ls * per_sector + rem;
        const int shift = have ? (int)(rem / J.chunks) : 0;
        const long long chunk = have ? rem - (long long)shift * J.chunks : 0;
        const int psec = J.sector_begin + ls;
        if (s_abort) { /* the pass was stopped: its remaining items contribute nothing */
            if (have && tl < J.n_slots * 2) J.partials[local * J.n_slots * 2 + tl] = 0.0;
            if (have && tl == 0) J.part_fails[local] = 0;
            __syncthreads();
            continue;
        }
        int level = -1; /* island level: the FP64 kernel has evaluated the island points and written the partial */
        if (J.sector_prec) {
            const PackedSector *gps = reinterpret_cast<const PackedSector *>(J.packed + J.sectors_off) + psec;
            const int code = J.sector_prec[gps->orig_index];
            level = island_level(code);
            if (code != 1 && level < 0) {
                __syncthreads();
                continue;
            }
        }
        if (psec != cur || jb != cur_job) {
            stage_sector_f2(J.packed, J.sectors_off, J.termsf_off, psec, smem);
            __syncthreads();
            cur = psec;
            cur_job = jb;
        }
        const Exps ex = Pol::exps(J);
        const Pol pol = Pol::make(T, sec, psec);
        const uint32_t n = J.n;
        const float invnf = 1.f / (float)n;
        const float lam = (float)J.lambda[sec.orig_index];
        uint32_t rj[S], aj[S], zs[S];
        float bj[S];
        const long long i0 = chunk * (long long)stride * jt.P + tl;
#pragma unroll
        for (int j = 0; j < S; ++j) {
            split_shift(J.shifts[6 * shift + j], n, aj[j], bj[j]);
            rj[j] = (uint32_t)(((unsigned long long)i0 * J.z[j]) % n);
            zs[j] = J.zstep[j];
        }
        float acc[2 * (MAXM + 1)], cmp[2 * (MAXM + 1)];
#pragma unroll
        for (int q = 0; q < 2 * (MAXM + 1); ++q) acc[q] = cmp[q] = 0.f;
        uint32_t fails = 0;
        const float rn = island_rn(n), xi = island_xi(level < 0 ? 0 : level);
        const int M = sec.M, sigma = sec.sigma;
        const unsigned smask = (unsigned)sec.sing_mask;
        for (int p0 = 0; p0 < jt.P; p0 += 2 * jt.pairs) {
            unsigned lives = 0; /* two bits per pair */
            float2 w0 = bc2(0.f), w1 = bc2(0.f); /* weights of the (at most two) pairs */
            unsigned Y = 0, count = 0;
            do {
                const unsigned next = (Y - smask) & smask;
                for (int q = 0; q < jt.pairs && p0 + 2 * q < jt.P; ++q) {
                    float2 t[S], tm[S];
                    if (Y == 0) {
                        bool live[2];
                        float2 x[S], y[S], w;
                        next_pair<S>(i0, p0 + 2 * q, jt.P, stride, n, invnf, level, smask, rn, xi, rj, aj, bj, zs, live, x, y);
                        live[0] = live[0] && have;
                        live[1] = live[1] && have;
                        if (!(live[0] || live[1]) || !pair_setup<S>(x, y, jt.r, live, t, tm, w)) continue;
                        lives |= (live[0] ? 1u : 0u) << (2 * q) | (live[1] ? 2u : 0u) << (2 * q);
#pragma unroll
                        for (int j = 0; j < S; ++j) st(q, PS::T + j) = t[j];
                        if (smask) {
#pragma unroll
                            for (int j = 0; j < S; ++j) st(q, PS::TM + j) = tm[j];
                        }
                        if (q == 0) w0 = w;
                        else w1 = w;
                    } else {
                        if (!((lives >> (2 * q)) & 3u)) continue;
#pragma unroll
                        for (int j = 0; j < S; ++j) {
                            const bool zj = (Y >> j) & 1u;
                            t[j] = zj ? bc2(0.f) : st(q, PS::T + j);
                            tm[j] = zj ? bc2(1.f) : st(q, PS::TM + j);
                        }
                    }
                    float2 d[S];
                    c2 detJ;
                    deform_f2<S>(pol, Y, t, tm, lam, d, detJ);
#pragma unroll
                    for (int j = 0; j < S; ++j) st(q, PS::D + j) = d[j];
                    st(q, PS::DET) = detJ.re;
                    st(q, PS::DET + 1) = detJ.im;
                }
                __syncthreads();
                for (int q = 0; q < jt.pairs && p0 + 2 * q < jt.P; ++q) {
                    const unsigned lv = (lives >> (2 * q)) & 3u;
                    if (!lv) continue;
                    const bool live[2] = {(lv & 1u) != 0, (lv & 2u) != 0};
                    float2 t[S], tt[S], d[S];
#pragma unroll
                    for (int j = 0; j < S; ++j) {
                        t[j] = st(q, PS::T + j);
                        tt[j] = (Y >> j) & 1u ? bc2(0.f) : t[j];
                        d[j] = st(q, PS::D + j);
                    }
                    const int need = M - sigma + __popc(count);
                    c2 G0, X;
                    value_f2<S>(sec, pol, Y, tt, d, c2{st(q, PS::DET), st(q, PS::DET + 1)}, MAXM > 0 && need > 0, ex, live, G0, X,
                                fails);
                    c2 o[MAXM + 1];
#pragma unroll
                    for (int m = 0; m <= MAXM; ++m)
                        o[m] = count == 0 ? zero_c2() : c2{st(q, PS::O + 2 * m), st(q, PS::O + 2 * m + 1)};
                    float2 one[MAXM + 1], Lt[S], a[S][MAXM + 1];
#pragma unroll
                    for (int m = 0; m <= MAXM; ++m) one[m] = bc2(m == 0 ? 1.f : 0.f);
                    pair_series<S, MAXM>(sec, t, Lt, a);
                    subset_add2<MAXM>(M, o, G0, X, one, 0, sigma, count, a, need);
                    if (next != 0) {
#pragma unroll
                        for (int m = 0; m <= MAXM; ++m) {
                            st(q, PS::O + 2 * m) = o[m].re;
                            st(q, PS::O + 2 * m + 1) = o[m].im;
                        }
                    } else {
                        const float2 w = q == 0 ? w0 : w1;
#pragma unroll
                        for (int m = 0; m <= MAXM; ++m) o[m] = cscale2(o[m], w);
                        add_pair<MAXM>(acc, cmp, o, live);
                    }
                }
                ++count;
                Y = next;
            } while (Y != 0);
        }
        warp_sums<MAXM>(acc, cmp, fails, s_red[warp], &s_fail[warp]);
        __syncthreads();
        if (have && tl < 32) write_partial<MAXM>(J, local, tl, s_red + group * nwarps, s_fail + group * nwarps, nwarps, level >= 0);
        __syncthreads();
    }
}

/* ------------------------------------------------------------------ K3: FP32-versus-FP64 probe per sector
 * One thread-block cluster per sector (cluster size = the launch's cluster dimension, 1 when clusters cannot be
 * had): block r of the cluster takes the sample points k = r * blockDim + thread (+ blockDim * cluster size), each
 * block reduces its threads in fixed order into shared memory, and block 0 adds the blocks' totals in rank order
 * through distributed shared memory -- deterministic, and no scratch in global memory. */
DEV unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
DEV unsigned cluster_blocks() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
/* every thread of every block of the cluster; orders the cluster's shared-memory writes before later reads */
DEV void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
/* a double in the shared memory of block `rank` of this cluster, at the address of `p` in this block */
DEV double ld_cluster(const double *p, unsigned rank) {
    const unsigned local = (unsigned)__cvta_generic_to_shared(p);
    unsigned remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(remote) : "memory");
    return v;
}

template <int S, bool DEF, int MAXM, class Pol>
DEV void probe_body(const ProbeArgs &a) {
    extern __shared__ __align__(16) unsigned char smem[];
    /* per bin: points, then per slot sum |e|, sum e re, sum e im, sum |e|^2 (e = v32 - v64) */
    constexpr int NBIN = 1 + 4 * (MAXM + 1);
    constexpr int NB = QMC_ISLAND_BINS * NBIN;
    constexpr int NA = 4 * (MAXM + 1);
    __shared__ double s_red[4][NA + NB];
    __shared__ double s_tot[NA + NB];
    const unsigned crank = cluster_rank(), csize = cluster_blocks();
    const int psec = a.sector_begin + (int)(blockIdx.x / csize);
    logtab_init();
    /* FP64 record + terms, then the FP32 terms */
    stage_sector(a.packed, a.sectors_off, a.terms_off, psec, smem);
    const PackedSector *gps = reinterpret_cast<const PackedSector *>(a.packed + a.sectors_off) + psec;
    const int nt = gps->n_terms;
    unsigned char *smf = smem + sizeof(PackedSector) + (size_t)nt * sizeof(PackedTerm);
    {
        const int4 *tsrc = reinterpret_cast<const int4 *>(a.packed + a.termsf_off) + gps->term0;
        int4 *tdst = reinterpret_cast<int4 *>(smf);
        for (int k = threadIdx.x; k < nt; k += blockDim.x) tdst[k] = tsrc[k];
    }
    __syncthreads();
    const PackedSector &sec = *reinterpret_cast<const PackedSector *>(smem);
    const PackedTerm *T = reinterpret_cast<const PackedTerm *>(smem + sizeof(PackedSector));
    const PackedTermF *TF = reinterpret_cast<const PackedTermF *>(smf);
    const Pol pol = Pol::make(TF, sec, psec);
    const Exps ex{a.eU0, a.eU1, a.eF0, a.eF1};
    const double lam = a.lambda[sec.orig_index];
    const float invnf = 1.f / (float)a.n;
    const unsigned long long stride = a.n_sample >= (int64_t)a.n ? 1ull : (unsigned long long)(a.n / a.n_sample);
    double acc[NA];
#pragma unroll
    for (int q = 0; q < NA; ++q) acc[q] = 0.0;
    double bacc[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) bacc[q] = 0.0;
    const float rn = island_rn(a.n);
    uint32_t Rj[S], aj[S];
    float bj[S];
#pragma unroll
    for (int j = 0; j < S; ++j) {
        Rj[j] = wrap_threshold(a.shift[j], a.n, a.invn);
        split_shift(a.shift[j], a.n, aj[j], bj[j]);
    }
    uint32_t f64 = 0, f32 = 0;
    const long long step = (long long)blockDim.x * csize;
    for (long long k = (long long)crank * blockDim.x + threadIdx.x;
         k < a.n_sample && (unsigned long long)k * stride < a.n; k += step) {
        const unsigned long long i = (unsigned long long)k * stride;
        double x[S];
        float xf[S], yf[S];
        uint32_t kk[S];
#pragma unroll
        for (int j = 0; j < S; ++j) {
            const uint32_t r = (uint32_t)((i * a.z[j]) % a.n);
            x[j] = fma((double)r, a.invn, a.shift[j]) - (r >= Rj[j] ? 1.0 : 0.0);
            lattice_f32(r, aj[j], bj[j], a.n, invnf, xf[j], yf[j]);
            kk[j] = shifted_index(r, aj[j], a.n);
        }
        const int bin = island_bin(island_key<S>(kk, (unsigned)sec.sing_mask, rn));
        cd v64[MAXM + 1];
        cf v32[MAXM + 1];
        point_integrand<S, DEF, MAXM>(sec, TabPol<S>{T, &sec}, x, a.r, lam, ex, v64, f64);
        point_integrand_f<S, DEF, MAXM>(sec, pol, xf, yf, a.r, (float)lam, ex, v32, f32);
#pragma unroll
        for (int b = 0; b < QMC_ISLAND_BINS; ++b) {
            if (b != bin) continue;
            bacc[b * NBIN] += 1.0;
        }
#pragma unroll
        for (int n = 0; n <= MAXM; ++n) {
            const double dr = (double)v32[n].x - v64[n].x, di = (double)v32[n].y - v64[n].y;
            const double m = hypot(dr, di);
            acc[4 * n] += hypot(v64[n].x, v64[n].y);
            acc[4 * n + 1] += m;
            acc[4 * n + 2] += dr;
            acc[4 * n + 3] += di;
#pragma unroll
            for (int b = 0; b < QMC_ISLAND_BINS; ++b) {
                if (b != bin) continue;
                double *e = &bacc[b * NBIN + 1 + 4 * n];
                e[0] += m;
                e[1] += dr;
                e[2] += di;
                e[3] = fma(m, m, e[3]);
            }
        }
    }
    /* threads -> warps (shuffle tree) -> block (warps in order) -> cluster (blocks in rank order) */
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = (int)(blockDim.x >> 5);
#pragma unroll
    for (int q = 0; q < NA + NB; ++q) {
        double v = q < NA ? acc[q] : bacc[q - NA];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) s_red[warp][q] = v;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < NA + NB; q += blockDim.x) {
        double v = 0.0;
        for (int w = 0; w < nwarps; ++w) v += s_red[w][q];
        s_tot[q] = v;
    }
    cluster_sync_all();
    if (crank == 0) {
        for (int q = threadIdx.x; q < 4 * a.n_slots; q += blockDim.x) {
            double v = 0.0;
            if (q < NA)
                for (unsigned r = 0; r < csize; ++r) v += ld_cluster(&s_tot[q], r);
            a.out[(size_t)sec.orig_index * a.n_slots * 4 + q] = v;
        }
        if (a.bins) {
            const int per = QMC_ISLAND_BIN_WORDS(a.n_slots);
            for (int q = threadIdx.x; q < QMC_ISLAND_BINS * per; q += blockDim.x) {
                const int b = q / per, e = q - b * per; /* e = 0: points; 1 + 4 slot + {0,1,2,3}: errors */
                double v = 0.0;
                if (e < NBIN)
                    for (unsigned r = 0; r < csize; ++r) v += ld_cluster(&s_tot[NA + b * NBIN + e], r);
                a.bins[(size_t)sec.orig_index * QMC_ISLAND_BINS * per + q] = v;
            }
        }
    }
    /* the other blocks keep their shared memory until block 0 has read it */
    cluster_sync_all();
}

template <int S, bool DEF, int MAXM>
__global__ void __launch_bounds__(128) qmc_probe_kernel(ProbeArgs a) {
    probe_body<S, DEF, MAXM, TabPolF<S>>(a);
}

/* ------------------------------------------------------------------ per-point values on explicit indices */
template <int S, int MAXM>
__global__ void __launch_bounds__(256) qmc_points_kernel_taylor(PointArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    logtab_init();
    stage_sector(a.packed, a.sectors_off, a.terms_off, a.sector, smem);
    __syncthreads();
    const PackedSector &sec = *reinterpret_cast<const PackedSector *>(smem);
    const PackedTerm *T = reinterpret_cast<const PackedTerm *>(smem + sizeof(PackedSector));
    const Exps ex{a.eU0, a.eU1, a.eF0, a.eF1};
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < a.npts;
         j += (long long)gridDim.x * blockDim.x) {
        const unsigned long long i = (unsigned long long)a.idx[j];
        double x[S];
#pragma unroll
        for (int d = 0; d < S; ++d) {
            const uint32_t rj = (uint32_t)((i * a.z[d]) % a.n);
            const double v = fma((double)rj, a.invn, a.shift[d]);
            x[d] = v >= 1.0 ? v - 1.0 : v;
        }
        double val[MAXM + 1];
        point_integrand_taylor<S, MAXM>(sec, T, x, a.r, ex, val);
        for (int n = 0; n < a.n_slots; ++n) {
            a.out[(j * a.n_slots + n) * 2] = n <= MAXM ? val[n < MAXM + 1 ? n : 0] : 0.0;
            a.out[(j * a.n_slots + n) * 2 + 1] = 0.0;
        }
        a.fails[j] = 0;
    }
}

template <int S, bool DEF, int MAXM>
__global__ void __launch_bounds__(256) qmc_points_kernel(PointArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    logtab_init();
    stage_sector(a.packed, a.sectors_off, a.terms_off, a.sector, smem);
    __syncthreads();
    const PackedSector &sec = *reinterpret_cast<const PackedSector *>(smem);
    const PackedTerm *T = reinterpret_cast<const PackedTerm *>(smem + sizeof(PackedSector));
    const Exps ex{a.eU0, a.eU1, a.eF0, a.eF1};
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < a.npts;
         j += (long long)gridDim.x * blockDim.x) {
        const unsigned long long i = (unsigned long long)a.idx[j];
        double x[S];
#pragma unroll
        for (int d = 0; d < S; ++d) {
            const uint32_t rj = (uint32_t)((i * a.z[d]) % a.n);
            const double v = fma((double)rj, a.invn, a.shift[d]);
            x[d] = v >= 1.0 ? v - 1.0 : v;
        }
        cd val[MAXM + 1];
        uint32_t f = 0;
        point_integrand<S, DEF, MAXM>(sec, TabPol<S>{T, &sec}, x, a.r, a.lambda, ex, val, f);
        for (int n = 0; n < a.n_slots; ++n) {
            const cd v = n <= MAXM ? val[n < MAXM + 1 ? n : 0] : mk(0.0, 0.0);
            a.out[(j * a.n_slots + n) * 2] = v.x;
            a.out[(j * a.n_slots + n) * 2 + 1] = v.y;
        }
        a.fails[j] = (int32_t)f;
    }
}
