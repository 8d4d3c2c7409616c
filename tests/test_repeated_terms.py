"""Tables that list a monomial more than once (`qmc_prepare` takes them; the coefficients add up): the generated code
holds every such term, in both precisions, and is written in finite time."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

import workloads as W
from paper_1508_02512_gb300 import _native as N
from paper_1508_02512_gb300 import api
from paper_1508_02512_gb300 import tables as T
from test_generated_source import TERM_D, blocks, host_harness64, image, subsets

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WORK = os.path.join(ROOT, "tests", "_gen_build")


def table(cfg, which, k):
    """cfg's table with term k of U~ or F~ (k = -1: every term) of every sector written as a quarter and, at the end of
    the list, three quarters: both parts and their sum are exact in FP64 and FP32 alike"""
    meta, leaves = T.read_table(T.compile_integral(cfg.topology, T.zero_invariants_of(cfg.topology, cfg.point)))
    for s in leaves:
        P = getattr(s, which)
        rows = np.arange(len(P.e)) if k < 0 else np.array([k % len(P.e)])
        c = P.c.copy()
        c[rows] *= 0.25
        setattr(s, which, T.Poly(np.concatenate([P.e, P.e[rows]]), np.concatenate([c, 0.75 * P.c[rows]])))
    return T.write_table(leaves, meta)


SPLITS = [("F", 0), ("F", -1), ("U", 0), ("U", -1)]


@pytest.mark.parametrize("which,k", SPLITS)
@pytest.mark.parametrize("cfg", [W.CONFIG0, W.CONFIG1], ids=lambda c: c.name)
def test_source_is_generated_and_holds_every_term(cfg, which, k):
    """In a process of its own with a time limit (a second is ample), then each FP64 function against the table's terms
    summed with numpy: both are a few dozen additions and products, 1e-14 of the summed magnitudes."""
    code = ("import sys; sys.path[:0] = [%r, %r]; import workloads as W, test_repeated_terms as R; from paper_1508_02512_gb300 "
            "import api; c = W.%s; p = api.prepare(R.table(c, %r, %d), c.kin, c.order_min, c.order_max); "
            "[api.gen_source(p, q) for q in (0, 1)]" % (ROOT, os.path.dirname(os.path.abspath(__file__)),
                                                        "CONFIG0" if cfg is W.CONFIG0 else "CONFIG1", which, k))
    assert subprocess.run([sys.executable, "-c", code], timeout=120).returncode == 0
    prep = api.prepare(table(cfg, which, k), cfg.kin, cfg.order_min, cfg.order_max)
    h, secs, _ = image(prep)
    terms = np.frombuffer(bytes(prep.packed), dtype=TERM_D, count=h.n_terms_total, offset=h.terms_off)
    os.makedirs(WORK, exist_ok=True)
    stem = os.path.join(WORK, f"rep_{cfg.name}_{which}{k}")
    with open(stem + ".cpp", "w") as f:
        f.write(host_harness64(api.gen_source(prep, N.QMC_PREC_FP64), h, secs))
    subprocess.check_call(["g++", "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-o", stem + ".so", stem + ".cpp"])
    L = ctypes.CDLL(stem + ".so")
    S = h.dim
    rng = np.random.Generator(np.random.PCG64(3))

    def ptr(a):
        return a.ctypes.data_as(ctypes.c_void_p)

    for i, s in enumerate(secs):
        Ts = np.ascontiguousarray(terms[s.term0: s.term0 + s.n_terms])
        U, F, G, H = blocks(h, s)
        for Y in subsets(s.sing_mask):
            t = rng.uniform(0.0, 1.0, S)
            t[[j for j in range(S) if (Y >> j) & 1]] = 0.0
            if s.kind != 2:
                out = np.zeros(2)
                L.h_ufr(i, Y, ptr(Ts), ptr(t), ptr(out))
                want, x = [U, F], [t, t]
                got = list(out)
            else:
                g, hh, uf = np.zeros(S), np.zeros(S * (S + 1) // 2), np.zeros(4)
                z = t * (1 - 0.3j * rng.uniform(0, 1, S))
                L.h_gh(i, Y, ptr(Ts), ptr(t), ptr(g), ptr(hh))
                L.h_ufc(i, Y, ptr(Ts), ptr(np.ascontiguousarray(np.stack([z.real, z.imag], -1))), ptr(uf))
                want, x = G + H + [U, F], [t] * (S + len(hh)) + [z, z]
                got = list(g) + list(hh) + [complex(uf[0], uf[1]), complex(uf[2], uf[3])]
            for (lo, hi), xv, gv in zip(want, x, got):
                parts = [tt["c"] * np.prod(xv ** tt["e"][:S]) for tt in Ts[lo:hi]]
                assert abs(gv - sum(parts)) <= 1e-14 * sum(abs(p) for p in parts), (i, Y)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [N.QMC_PREC_FP64, N.QMC_PREC_MIXED], ids=["fp64", "mixed"])
def test_pass_equals_that_of_the_plain_table(precision):
    """The same integral, so the same sums to the rounding of the polynomials: FP64 1e-12 of a sector's largest sum (as in
    the parity tests), FP32 1e-5 (some hundred roundings of 6e-8)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = W.CONFIG1
    n, z = api.builtin_lattices()[0]
    sums = []
    for blob in (T.compile_integral(cfg.topology, T.zero_invariants_of(cfg.topology, cfg.point)), table(cfg, "F", -1)):
        prep = api.prepare(blob, cfg.kin, cfg.order_min, cfg.order_max)
        dev = api.DeviceIntegral(prep)
        p = api.make_pass(n, z, 4, 3, precision)
        out, fails = dev.outputs(p)
        lam = torch.full((prep.info.n_sectors,), 0.5, dtype=torch.float64, device="cuda")
        dev.eval_sums(p, torch.tensor(W.shifts(2, 4), device="cuda"), lam, out, fails)
        torch.cuda.synchronize()
        sums.append(out.cpu().numpy())
    scale = np.abs(sums[0]).max(axis=(1, 2, 3), keepdims=True)
    assert np.isfinite(sums[1]).all()
    assert (np.abs(sums[1] - sums[0]) <= (1e-12 if precision == N.QMC_PREC_FP64 else 1e-5) * scale).all()
