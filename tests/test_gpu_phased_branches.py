"""The phased FP32 kernel (deformed sectors of five and six dimensions) in all its forms: five dimensions, series of one,
three and five slots (with five, one pair of points per thread fits in six dimensions), sectors in FP64, in FP32 and in FP32
with FP64 islands side by side, several passes in one launch, and a stopped pass among them.

The integrals are sixteen sectors of the non-planar double box; the five-dimensional table is theirs with the last variable
set to 1 (a table like any other to the library).

Sums are held against the FP64 pass on the same points, sector by sector and slot by slot.  The probe evaluates every point
of the first shift in both precisions and gives sum |v64| and sum |v32 - v64|: the difference of the sums is bounded by the
latter, up to the rounding of the code that made v32 (generated here, table-driven in the probe: as large, so a factor 4)."""
import ctypes

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1508_02512_gb300 import _native as N  # noqa: E402
from paper_1508_02512_gb300 import api  # noqa: E402
from paper_1508_02512_gb300 import tables as T  # noqa: E402

LAM, N_POINTS = 0.1, 1021
cache = {}


def integral(dim, order_max):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if (dim, order_max) not in cache:
        cfg = W.CONFIG3
        meta, leaves = T.read_table(T.compile_integral(cfg.topology, T.zero_invariants_of(cfg.topology, cfg.point)))
        by_poles = sorted(leaves, key=lambda s: int(np.sum(s.A == -1)))
        leaves = [s for k in (0, len(leaves) // 3, len(leaves) // 2, -4) for s in by_poles[k:][:4]]
        if dim == 5:
            meta = dict(meta, dim=5, nu=[1] * 6, n_nu=6, eU=(0, 3), eF=(2, 2))
            for s in leaves:
                s.A, s.B = s.A[:5], s.B[:5]
                s.U, s.F = T.Poly(s.U.e[:, :5], s.U.c).simplified(), T.Poly(s.F.e[:, :5], s.F.c).simplified()
        prep = api.prepare(T.write_table(leaves, meta), cfg.kin, -2, order_max)
        assert all(prep.sector(k).kind == 2 for k in range(prep.info.n_sectors)) and prep.info.dim == dim
        cache[dim, order_max] = prep, api.DeviceIntegral(prep)
    return cache[dim, order_max]


def run(dim, order_max, prec, m=3, block=128, points=4, codes=None):
    prep, dev = integral(dim, order_max)
    z = [pow(76, j, N_POINTS) or 1 for j in range(6)]
    p = api.make_pass(N_POINTS, z, m, 3, prec, block=block, points_per_thread=points)
    keep = torch.tensor(codes, dtype=torch.int32, device="cuda") if codes is not None else None
    if keep is not None:
        p.sector_precision = keep.data_ptr()
    sh = torch.tensor(W.shifts(5, m), device="cuda")
    lam = torch.full((prep.info.n_sectors,), LAM, dtype=torch.float64, device="cuda")
    sums, fails = dev.outputs(p)
    dev.eval_sums(p, sh, lam, sums, fails)
    torch.cuda.synchronize()
    return sums.cpu().numpy(), fails.cpu().numpy()


def probed(dim, order_max):
    """per sector and slot: sum |v64| and sum |v32 - v64| over the points of the first shift"""
    prep, dev = integral(dim, order_max)
    z = [pow(76, j, N_POINTS) or 1 for j in range(6)]
    p = api.make_pass(N_POINTS, z, 3, 3, N.QMC_PREC_MIXED)
    out = torch.zeros((prep.info.n_sectors, prep.info.n_slots, 4), dtype=torch.float64, device="cuda")
    lam = torch.full((prep.info.n_sectors,), LAM, dtype=torch.float64, device="cuda")
    sh = torch.tensor(W.shifts(5, 3), device="cuda")
    N.check(N.lib().qmc_probe_precision(prep.packed, dev.dpacked.data_ptr(), ctypes.byref(p), sh.data_ptr(), lam.data_ptr(),
                                        4096, out.data_ptr(), None), "qmc_probe_precision")
    torch.cuda.synchronize()
    pr = out.cpu().numpy()
    return pr[..., 0], pr[..., 1]


FORMS = [(6, -2), (6, 0), (6, 2), (5, -2), (5, 0), (5, 2)]


@pytest.mark.parametrize("dim,order_max", FORMS)
def test_sums_against_fp64(dim, order_max):
    a, _ = run(dim, order_max, N.QMC_PREC_MIXED)
    b, _ = run(dim, order_max, N.QMC_PREC_FP64)
    mag, err = probed(dim, order_max)
    assert np.isfinite(a).all() and (mag[:, 0] > 0).all()
    d = np.hypot(*np.moveaxis(a[:, 0] - b[:, 0], -1, 0))
    assert (d <= 4 * err + 1e-7 * mag).all()


# a point left out or counted twice changes a sum by 1e-3 of it; shapes agree to the order of summation (as in the pass tests)
@pytest.mark.parametrize("dim,order_max", FORMS)
@pytest.mark.parametrize("block,points", [(96, 3), (32, 64), (128, 16)])
def test_sums_do_not_depend_on_the_launch_shape(dim, order_max, block, points):
    a, fa = run(dim, order_max, N.QMC_PREC_MIXED, block=block, points=points)
    b, fb = run(dim, order_max, N.QMC_PREC_MIXED)
    scale = np.abs(b).max(axis=(1, 2, 3), keepdims=True)
    assert (np.abs(a - b) <= 1e-11 * scale).all() and np.array_equal(fa, fb)


@pytest.mark.parametrize("codes", [(1, 1, 2, 3, 4, 5, 6, 7) * 2, (2, 0, 1, 0, 0, 3, 0, 2) * 2, (0,) * 15 + (3,)])
@pytest.mark.parametrize("dim,order_max", [(6, 0), (6, 2), (5, 0)])
def test_sectors_of_different_precision(dim, order_max, codes):
    a, fa = run(dim, order_max, N.QMC_PREC_MIXED, codes=codes)
    full, _ = run(dim, order_max, N.QMC_PREC_FP64)
    single, _ = run(dim, order_max, N.QMC_PREC_MIXED)
    mag, err = probed(dim, order_max)
    d = np.hypot(*np.moveaxis(a[:, 0] - full[:, 0], -1, 0))
    assert (d <= 4 * err + 1e-7 * mag).all()
    for s, code in enumerate(codes):
        if code == 0:
            assert np.array_equal(a[s], full[s])
        if code == 1:
            assert np.array_equal(a[s], single[s])
    for block, points in ((96, 3), (64, 5)):
        b, fb = run(dim, order_max, N.QMC_PREC_MIXED, block=block, points=points, codes=codes)
        scale = np.abs(a).max(axis=(1, 2, 3), keepdims=True)
        assert (np.abs(a - b) <= 1e-11 * scale).all() and np.array_equal(fa, fb)


def test_several_passes_in_one_launch_and_a_stopped_one():
    """Same kernel and shape, so one launch: each pass equals itself alone bit for bit; with the middle one's flag set its
    sums and counts are zero and the others are unchanged."""
    prep, dev = integral(6, 0)
    lam = torch.full((prep.info.n_sectors,), LAM, dtype=torch.float64, device="cuda")
    host = ctypes.create_string_buffer(prep.packed)
    items, keep, alone = (N.qmc_batch_item * 3)(), [], []
    for i, (n, m) in enumerate(((1021, 3), (4093, 2), (257, 5))):
        p = api.make_pass(n, [pow(76, j, n) or 1 for j in range(6)], m, 3, N.QMC_PREC_MIXED, block=96, points_per_thread=4)
        sh = torch.tensor(W.shifts(20 + i, m), device="cuda")
        sums, fails = dev.outputs(p)
        dev.eval_sums(p, sh, lam, sums, fails)
        torch.cuda.synchronize()
        alone.append((sums.clone(), fails.clone()))
        keep.append((p, sh, sums, fails))
        items[i].packed_host, items[i].packed_dev, items[i].pass_ = ctypes.addressof(host), dev.dpacked.data_ptr(), p
        items[i].shifts_dev, items[i].lambda_dev = sh.data_ptr(), lam.data_ptr()
        items[i].sums_dev, items[i].fails_dev = sums.data_ptr(), fails.data_ptr()
    need = N.lib().qmc_batch_scratch_bytes(items, 3)
    scratch = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
    base = scratch.data_ptr() + (-scratch.data_ptr()) % 256
    stop = torch.ones(1, dtype=torch.int32, device="cuda")
    for stopped in (None, 1):
        if stopped is not None:
            items[stopped].abort_flag = stop.data_ptr()
        for _, _, sums, fails in keep:
            sums.fill_(7.0)
            fails.fill_(7)
        N.check(N.lib().qmc_eval_batch(items, 3, base, need, torch.cuda.current_stream().cuda_stream), "qmc_eval_batch")
        torch.cuda.synchronize()
        for i, (_, _, sums, fails) in enumerate(keep):
            if i == stopped:
                assert int(torch.count_nonzero(sums)) == 0 and int(torch.count_nonzero(fails)) == 0
            else:
                assert torch.equal(sums, alone[i][0]) and torch.equal(fails, alone[i][1])
