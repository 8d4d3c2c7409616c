"""The library's choice of points per thread (`default_points` in csrc/qmc_pass.cpp), cut out and compiled for the host, and
what does not depend on it: with the shape given, the sums of a shift are the same whatever other shifts the pass holds."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import workloads as W
from paper_1508_02512_gb300 import _native as N
from paper_1508_02512_gb300 import api
from paper_1508_02512_gb300 import tables as T

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WORK = os.path.join(ROOT, "tests", "_gen_build")
CSRC = os.path.join(ROOT, "paper_1508_02512_gb300", "csrc")


@pytest.fixture(scope="module")
def points():
    text = open(os.path.join(CSRC, "qmc_pass.cpp")).read()
    i = text.index("int default_points(const PackedHeader *h, const qmc_pass *p, int block) {")
    body = text[i:text.index("\n}\n", i) + 3]
    os.makedirs(WORK, exist_ok=True)
    cpp, so = os.path.join(WORK, "launch_shape.cpp"), os.path.join(WORK, "launch_shape.so")
    with open(cpp, "w") as f:
        f.write('#include <cstring>\n#include "qmc_internal.h"\n' + body + r'''
extern "C" int h_points(int sectors, int precision, long n, int m, int block) {
    PackedHeader h;
    qmc_pass p;
    std::memset(&h, 0, sizeof(h));
    std::memset(&p, 0, sizeof(p));
    h.n_sectors = sectors;
    p.precision = precision;
    p.lattice.n = n;
    p.n_shifts = m;
    return default_points(&h, &p, block);
}
''')
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, cpp, "-o", so], check=True)
    f = ctypes.CDLL(so).h_points
    return lambda s, prec, n, m, b: f(s, prec, ctypes.c_long(n), m, b)


F, M = N.QMC_PREC_FP64, N.QMC_PREC_MIXED


@pytest.mark.parametrize("sectors,precision,n,m,block,want", [
    (1, F, 1021, 912, 128, 8), (1, F, 1021, 911, 128, 4),          # 6 items per SM (152) and one item less
    (1, F, 1021, 76, 128, 4), (1, F, 1021, 75, 128, 2),            # then one item per SM and two items less
    (48, F, 1100, 10, 128, 5), (48, F, 1100, 9, 128, 3),           # two equal chunks of 5 x 128, halved and rounded up
    (48, F, 257, 1, 128, 1), (48, F, 4093, 16, 128, 8), (4, F, 2049, 8, 64, 4),
    (48, M, 3001, 16, 128, 12), (48, M, 1048573, 16, 128, 16),     # equal chunks; the whole number
    (48, M, 1025, 16, 128, 6), (48, M, 37, 1, 128, 2),             # 5 and 1, made even: points go in pairs
    (1, F, 2147483647, 4096, 32, 8),
])
def test_chosen_points(points, sectors, precision, n, m, block, want):
    assert points(sectors, precision, n, m, block) == want


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [F, M], ids=["fp64", "mixed"])
def test_sums_of_a_shift_do_not_depend_on_the_others(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = W.CONFIG3
    prep = api.prepare(T.compile_integral(cfg.topology, T.zero_invariants_of(cfg.topology, cfg.point)), cfg.kin,
                       cfg.order_min, cfg.order_max)
    dev = api.DeviceIntegral(prep)
    n, z = api.builtin_lattices()[0]
    shifts = W.shifts(6, 16)
    lam = torch.full((prep.info.n_sectors,), 0.3, dtype=torch.float64, device="cuda")

    def run(sh):
        p = api.make_pass(n, z, len(sh), 3, precision, block=128, points_per_thread=4)
        sums, fails = dev.outputs(p)
        dev.eval_sums(p, torch.tensor(np.ascontiguousarray(sh), device="cuda"), lam, sums, fails)
        torch.cuda.synchronize()
        return sums.cpu().numpy(), fails.cpu().numpy()

    whole, fw = run(shifts)
    for part in (slice(0, 1), slice(3, 8)):
        s, f = run(shifts[part])
        assert np.array_equal(s, whole[:, part]) and np.array_equal(f, fw[:, part])
