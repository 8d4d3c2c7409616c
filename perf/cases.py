"""Workloads on which this repository's speed is measured.

A case is one call that a program using the library makes, at one size: a pass of the hot path over a prepared
integral (`DeviceIntegral.eval_sums`), an integration to a requested accuracy (`Context.integrate`), or a batch of
requests through the serving loop (`Context.submit` / `Context.wait`).  The integrals, kinematic points and shift
counts are those of `workloads/`; lattices are the built-in ladder's where its size is asked for, and Korobov
vectors (1, a, a^2, ...) for the sizes in between that a program with lattices of its own brings along.

`exact` evaluates the same lattice sums in plain torch, in 64 bits, from the sector table alone.
"""
import ctypes
import functools
import itertools
import math
import struct

import numpy as np
import torch

import workloads as W
from paper_1508_02512_gb300 import _native as N
from paper_1508_02512_gb300 import api
from paper_1508_02512_gb300 import tables as T

# integral -> (workload, deformation parameter at which its sign check holds at the workload's point)
INTEGRALS = {
    "massless_box": (W.CONFIG0, 0.0),
    "massive_box": (W.CONFIG1, 0.5),
    "planar_dbox": (W.CONFIG2, 0.25),
    "nonplanar_dbox": (W.CONFIG3, 0.25),
    "massless_dbox": (W.PAPER_IB, 0.0),
}
PRECISION = {"fp64": N.QMC_PREC_FP64, "mixed": N.QMC_PREC_MIXED}


def listed():
    def one(name, integral, precision, n, shifts, do="pass", **more):
        return dict(name=name, do=do, integral=integral, precision=precision, n=n, shifts=shifts, r=3, **more)

    return [
        # the first rung of the ladder on a one-loop integral: what a quick look or a small request costs
        one("box0_fp64_small", "massless_box", "fp64", 1021, 4),
        # the one-loop box with double poles at its full lattice: an ordinary one-loop FP64 pass
        one("box0_fp64", "massless_box", "fp64", 65521, 8),
        # the physical one-loop box, FP64, deformed sectors without poles: a precise one-loop value
        one("mbox_fp64", "massive_box", "fp64", 262139, 16),
        # the same in mixed precision at a large lattice: the one-loop throughput case
        one("mbox_mixed", "massive_box", "mixed", 1048573, 16),
        # the paper's one-loop scan: 64 kinematic points to 1e-4 through the serving loop
        one("mbox_scan", "massive_box", "mixed", 64, 16, do="scan", tol=1e-4),
        # the non-planar double box in FP64: what the FP64 paths of a two-loop integration spend their time on
        one("np_fp64", "nonplanar_dbox", "fp64", 16381, 16),
        # a two-loop mixed pass low on the ladder, lattice of the caller's own: every integration starts there
        one("np_mixed_small", "nonplanar_dbox", "mixed", 3001, 16),
        # the benchmark's step: the two-loop mixed pass at production size
        one("np_mixed", "nonplanar_dbox", "mixed", 1048573, 16),
        # the whole call: the non-planar double box to 1e-3, lattices, precisions and lambda chosen by the library
        one("np_integrate", "nonplanar_dbox", "mixed", 0, 16, do="integrate", tol=1e-3),
        # the planar double box in mixed precision in the middle of the ladder, odd lattice size of the caller's own
        one("pl_mixed", "planar_dbox", "mixed", 50021, 16),
        # the massless double box with four poles (undeformed, up to 16 subtraction subsets per point) in FP64
        one("ib_fp64", "massless_dbox", "fp64", 8191, 16),
        # the same in mixed precision with the sector precisions the library picks for 1e-4 (FP64 islands, FP64 sectors)
        one("ib_mixed", "massless_dbox", "mixed", 65521, 16, tol=1e-4),
    ]


# largest lattice x shifts of a drawn pass, so that none costs more than the largest listed case
LARGEST = {
    ("massless_box", "fp64"): 6.0e6, ("massless_box", "mixed"): 6.0e7,
    ("massive_box", "fp64"): 1.6e7, ("massive_box", "mixed"): 1.6e8,
    ("planar_dbox", "fp64"): 3.0e5, ("planar_dbox", "mixed"): 1.2e7,
    ("nonplanar_dbox", "fp64"): 3.0e5, ("nonplanar_dbox", "mixed"): 1.2e7,
    ("massless_dbox", "fp64"): 3.0e5, ("massless_dbox", "mixed"): 1.0e6,
}


def draw(rng):
    """A pass of any of the integrals in either precision: small, ordinary and large lattices, ladder sizes and others."""
    integral, precision = rng.choice(sorted(LARGEST))
    shifts = rng.choice([1, 3, 4, 8, 16, 16, 20, 32])
    top = max(2000.0, min(4.0e6, LARGEST[integral, precision] / shifts))
    n = int(round(math.exp(rng.uniform(math.log(900.0), math.log(top)))))
    if rng.random() < 0.4:  # a rung of the built-in ladder
        n = max((ln for ln, _ in api.builtin_lattices() if ln <= n), default=1021)
    case = dict(do="pass", integral=integral, precision=precision, n=n, shifts=shifts, r=rng.choice([1, 2, 3, 3, 3]))
    if precision == "mixed" and integral == "massless_dbox":
        case["tol"] = rng.choice([1e-3, 1e-4])
    return case


# ---------------------------------------------------------------------------------------------- what a user holds
@functools.lru_cache(maxsize=None)
def table(integral):
    """The integral's sector table: compiled once, offline work for a user."""
    cfg = INTEGRALS[integral][0]
    return T.compile_integral(cfg.topology, T.zero_invariants_of(cfg.topology, cfg.point), strategy=cfg.strategy)


@functools.lru_cache(maxsize=None)
def scan_table():
    box = W.box(True)
    return T.compile_integral(box, T.zero_invariants_of(box, W.paper_ia_point(W.PAPER_IA_S_RANGE_GEV2[0])))


def vector(n):
    z = dict(api.builtin_lattices()).get(n)
    return z if z is not None else [pow(76, j, n) or 1 for j in range(6)]


def prepare(case, seed):
    cfg, lam = INTEGRALS[case["integral"]]
    prec = PRECISION[case["precision"]]
    if case["do"] == "pass":
        prep = api.prepare(table(case["integral"]), cfg.kin, cfg.order_min, cfg.order_max)
        api.gen_compile(prep, precision=prec)
        dev = api.DeviceIntegral(prep, "cuda")
        p = api.make_pass(case["n"], vector(case["n"]), case["shifts"], case["r"], prec)
        sh = torch.tensor(W.shifts(seed, case["shifts"]), device="cuda")
        lams = torch.full((prep.info.n_sectors,), lam, dtype=torch.float64, device="cuda")
        state = dict(do="pass", dev=dev, p=p, sh=sh, lam=lams)
        if "tol" in case:  # the precision of each sector, as an integration to this accuracy picks it
            api.gen_compile(prep, precision=N.QMC_PREC_FP64)
            state["codes"] = codes = precision_codes(prep, dev, p, sh, lams, case["tol"])
            p.sector_precision = codes.data_ptr()
        state["sums"], state["fails"] = dev.outputs(p)
        dev.scratch(p)
        return state
    ctx = api.Context(0, 4 << 30)
    if case["do"] == "integrate":
        blob, prep = table(case["integral"]), None
        iid = ctx.load_sectors(blob)
        ctx.set_kinematics(iid, cfg.kin, cfg.order_min, cfg.order_max)
        prep = api.prepare(blob, cfg.kin, cfg.order_min, cfg.order_max)
        state = dict(do="integrate", ctx=ctx, iid=iid, seed=seed, tol=case["tol"], shifts=case["shifts"], prec=prec)
    else:
        blob, topo = scan_table(), W.box(True)
        lo, hi = W.PAPER_IA_S_RANGE_GEV2
        s_vals = np.random.Generator(np.random.PCG64(seed)).uniform(lo, hi, case["n"])
        kin = [W.kinematics(topo, **W.paper_ia_point(s)) for s in s_vals]
        prep = api.prepare(blob, kin[0], 0, 0)
        state = dict(do="scan", ctx=ctx, iid=ctx.load_sectors(blob), kin=kin, seed=seed, tol=case["tol"],
                     shifts=case["shifts"], prec=prec)
    for pr in (N.QMC_PREC_FP64, prec):
        api.gen_compile(prep, precision=pr)
    return state


def precision_codes(prep, dev, p, sh, lam, tol):
    """qmc_probe_islands and qmc_choose_precision, as before the first FP32 pass of an integration."""
    ns, slots = prep.info.n_sectors, prep.info.n_slots
    out = torch.zeros((ns, slots, 4), dtype=torch.float64, device="cuda")
    bins = torch.zeros((ns, N.QMC_ISLAND_BINS, N.island_bin_words(slots)), dtype=torch.float64, device="cuda")
    N.check(N.lib().qmc_probe_islands(prep.packed, dev.dpacked.data_ptr(), ctypes.byref(p), sh.data_ptr(),
                                      lam.data_ptr(), 4096, out.data_ptr(), bins.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream), "qmc_probe_islands")
    pr, bn = out.cpu().numpy(), bins.cpu().numpy()
    codes = np.zeros(ns, dtype=np.int32)
    N.check(N.lib().qmc_choose_precision(prep.packed, 0, None, None, pr.ctypes.data, bn.ctypes.data, 4096, tol, 0.1,
                                         codes.ctypes.data, None), "qmc_choose_precision")
    return torch.from_numpy(codes).cuda()


def run(state):
    if state["do"] == "pass":
        state["dev"].eval_sums(state["p"], state["sh"], state["lam"], state["sums"], state["fails"])
        return {"sums": state["sums"], "fails": state["fails"]}
    ctx, iid = state["ctx"], state["iid"]
    more = dict(rel_tol=state["tol"], n_shifts=state["shifts"], lam=0.5, precision=state["prec"])
    if state["do"] == "integrate":
        value, error = api.result_arrays(ctx.integrate(iid, seed=state["seed"], **more))
        return {"value": value, "error": error}
    ids = [ctx.submit(iid, k, 0, 0, seed=state["seed"] + i, **more) for i, k in enumerate(state["kin"])]
    got = [api.result_arrays(ctx.wait(i)) for i in ids]
    return {"value": np.concatenate([v for v, _ in got]), "error": np.concatenate([e for _, e in got])}


# ---------------------------------------------------------------------------------------------- work and values
# evaluations of the whole calls (they depend on the seed; these are what they come to)
EVALS = {"integrate": 2.0e8, "scan": 2.8e5}


def work(case):
    """Floating-point work of the evaluations as the library counts it from the sector table (add, multiply 1, FMA 2);
    bytes: table, shifts, lambda in, sums and fail counts out."""
    cfg, _ = INTEGRALS[case["integral"]]
    blob = scan_table() if case["do"] == "scan" else table(case["integral"])
    kin = W.kinematics(W.box(True), **W.paper_ia_point(3.0e5)) if case["do"] == "scan" else cfg.kin
    info = api.prepare(blob, kin, cfg.order_min, cfg.order_max).info
    m, ns = case["shifts"], info.n_sectors
    io = info.packed_bytes + 48 * m + 8 * ns + ns * m * (16 * info.n_slots + 8)
    if case["do"] == "pass":
        return {"bytes": io, "flops": float(ns) * m * case["n"] * info.flops_per_eval}
    calls = case["n"] if case["do"] == "scan" else 1
    return {"bytes": calls * io, "flops": calls * EVALS[case["do"]] * info.flops_per_eval}


def read(blob):
    """The sector table: (powers of U and F, [(A, B, D, U, F)]), a polynomial as (exponents, coefficient rows)."""
    _, ns, dim, _, _, _, K, eU0, eU1, eF0, eF1, off = struct.unpack_from("<12i", blob, 8)
    sectors = []
    for _ in range(ns):
        nU, nF = struct.unpack_from("<2i", blob, off)
        AB = struct.unpack_from(f"<{2 * dim}i", blob, off + 8)
        off += 8 + 8 * dim
        (D,) = struct.unpack_from("<d", blob, off)
        off += 8
        polys = []
        for count in (nU, nF):
            rows = []
            for _ in range(count):
                rows.append((tuple(blob[off:off + dim]), struct.unpack_from(f"<{1 + K}d", blob, off + 8)))
                off += 16 + 8 * K
            polys.append(rows)
        sectors.append((AB[:dim], AB[dim:], D, polys[0], polys[1]))
    return (eU0, eU1, eF0, eF1), sectors


def polynomial(terms, var, zero=0):
    """sum c prod var_j^e_j over {exponents: c}; variables in the bit mask `zero` are zero."""
    memo = {}

    def mono(e):
        if e not in memo:
            j = max(k for k in range(len(e)) if e[k])
            rest = e[:j] + (e[j] - 1,) + e[j + 1:]
            memo[e] = mono(rest) * var[j] if any(rest) else var[j]
        return memo[e]

    acc = torch.zeros_like(var[0])
    for e, c in sorted(terms.items()):
        if any(e[j] and (zero >> j) & 1 for j in range(len(e))) or c == 0.0:
            continue
        acc = acc + (c * mono(e) if any(e) else c)
    return acc


def derivative(terms, j):
    return {e[:j] + (e[j] - 1,) + e[j + 1:]: c * e[j] for e, c in terms.items() if e[j]}


def transform(r, x):
    """phi_r(x) on [0, 1/2], its complement, and the weight phi_r'(x) (Eq. 21)."""
    u, lower = torch.minimum(x, 1.0 - x), x <= 0.5
    norm = math.factorial(2 * r + 1) / math.factorial(r) ** 2
    p = u * 0.0
    for i in range(r, -1, -1):
        p = p * u + norm * math.comb(r, i) * (-1) ** i / (r + i + 1)
    p = p * u ** (r + 1)
    return torch.where(lower, p, 1.0 - p), torch.where(lower, 1.0 - p, p), norm * (x * (1.0 - x)) ** r


def determinant(H, g, t, tm, lam):
    """det(dz/dt) of z = t - i lam t (1 - t) dF: complex symmetric elimination (similar matrix, Hermitian part 1)."""
    S, s = len(t), [torch.sqrt(a * b) for a, b in zip(t, tm)]
    M = {}
    for j in range(S):
        for k in range(j, S):
            b = s[j] * s[k] * H[j, k] + ((tm[j] - t[j]) * g[j] if j == k else 0.0)
            M[j, k] = torch.complex(torch.full_like(b, float(j == k)), -lam * b)
    det = 1.0
    for c in range(S):
        det = det * M[c, c]
        for j in range(c + 1, S):
            f = M[c, j] / M[c, c]
            for k in range(j, S):
                M[j, k] = M[j, k] - f * M[c, k]
    return det


def sector_values(powers, sector, inv, lam, r, x, slots):
    """w(x) x the sector's eps series at points x (Eqs. 9-12, 14): slot n is the coefficient of eps^(n - sigma)."""
    eU0, eU1, eF0, eF1 = powers
    A, B, D, U, F = sector
    S = len(A)
    Ut = {e: sum(a * b for a, b in zip(c, inv)) for e, c in U}
    Ft = {e: sum(a * b for a, b in zip(c, inv)) for e, c in F}
    signs = {math.copysign(1.0, c) for c in Ft.values() if c != 0.0}
    deformed = len(signs) == 2
    if signs == {-1.0}:
        Ft = {e: -c for e, c in Ft.items()}
    trio = [transform(r, x[j]) for j in range(S)]
    t, tm = [a for a, _, _ in trio], [a for _, a, _ in trio]
    w = functools.reduce(torch.mul, [a for _, _, a in trio])
    sing = [j for j in range(S) if A[j] == -1]
    M = len(sing)
    Lt = [torch.log(a) for a in t]
    out = [torch.zeros_like(w, dtype=torch.complex128 if deformed else torch.float64) for _ in range(slots)]
    dF = [derivative(Ft, j) for j in range(S)]
    for Y in itertools.chain.from_iterable(itertools.combinations(sing, k) for k in range(M + 1)):
        zero = sum(1 << j for j in Y)
        tt = [a * 0.0 if (zero >> j) & 1 else a for j, a in enumerate(t)]
        ttm = [a * 0.0 + 1.0 if (zero >> j) & 1 else a for j, a in enumerate(tm)]
        z, q, G = tt, None, D
        if deformed:
            g = [polynomial(dF[j], tt, zero) for j in range(S)]
            H = {(j, k): polynomial(derivative(dF[j], k), tt, zero) for j in range(S) for k in range(j, S)}
            G = D * determinant(H, g, tt, ttm, lam)
            q = [torch.complex(torch.ones_like(b), -lam * b * c) for b, c in zip(ttm, g)]
            z = [a * b for a, b in zip(tt, q)]
        u, f = polynomial(Ut, z, zero), polynomial(Ft, z, zero)
        G = G * u ** eU0 / f ** eF0
        X = eU1 * torch.log(u) - eF1 * torch.log(f) if M else None
        for j in range(S):
            if A[j] > 0:
                G = G * tt[j] ** A[j]
            if deformed and A[j] != 0:
                G = G * q[j] ** A[j]
            if M and B[j] != 0:
                if A[j] != -1:
                    X = X + B[j] * Lt[j]
                if deformed:
                    X = X + B[j] * torch.log(q[j])
        V = [torch.ones_like(w)] + [torch.zeros_like(w) for _ in range(M)]
        for j in sing:  # eps t^(-1 + B eps), and for a zeroed variable 1/B - eps t^(-1 + B eps)
            sign = -1.0 if j in Y else 1.0
            fj = [torch.full_like(w, 1.0 / B[j]) if j in Y else torch.zeros_like(w)]
            c = 1.0 / t[j]
            for n in range(1, M + 1):
                fj.append(sign * c)
                c = c * (B[j] * Lt[j]) / n
            V = [sum(V[k] * fj[n - k] for k in range(n + 1)) for n in range(M + 1)]
        term = G
        for n in range(M + 1):
            for k in range(M + 1 - n):
                out[n + k] = out[n + k] + term * V[k]
            if n < M:
                term = term * X / (n + 1)
    return [w * o for o in out]


def exact(case, seed):
    """The pass's sums in plain 64-bit torch; the fail counts are whole numbers and need no such value."""
    if case["do"] != "pass":
        return None
    cfg, lam = INTEGRALS[case["integral"]]
    powers, sectors = read(table(case["integral"]))
    n, m, r = case["n"], case["shifts"], case["r"]
    per_point = sum((1 << sum(a == -1 for a in A)) * (len(A) ** 2 * len(F) if len(A) > 3 else 100)
                    for A, _, _, _, F in sectors)
    if per_point * n * m > 2.0e11:  # more than about 20 seconds
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    inv = [1.0] + [float(v) for v in cfg.kin]
    sh = torch.tensor(W.shifts(seed, m), device=dev)
    z = vector(n)
    slots = 1 + max(sum(a == -1 for a in A) for A, _, _, _, _ in sectors)
    sums = torch.zeros((len(sectors), m, slots, 2), dtype=torch.float64, device=dev)
    step = max(1, (1 << 19) // n)  # shifts evaluated together
    for k0, i0 in itertools.product(range(0, m, step), range(0, n, 1 << 19)):
        i = torch.arange(i0, min(n, i0 + (1 << 19)), device=dev)
        d = sh[k0:k0 + step]
        x = [((i * z[j]) % n).double()[None, :] / n + d[:, j:j + 1] for j in range(len(sectors[0][0]))]
        x = [a - torch.floor(a) for a in x]
        for s, sector in enumerate(sectors):
            v = torch.stack([a.sum(dim=1) for a in sector_values(powers, sector, inv, lam, r, x, slots)], dim=1)
            v = v if v.is_complex() else torch.complex(v, torch.zeros_like(v))
            sums[s, k0:k0 + step] += torch.view_as_real(v)
    return {"sums": sums, "fails": None}
