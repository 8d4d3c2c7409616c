"""The phased FP32 kernel (deformed sectors of five and six dimensions): a block of 512 threads works on sets of items of
one sector, one item per group of `block` threads.  The point values do not depend on the launch shape, so passes with
other shapes, whose sets, groups, pairs and remainders differ, must give the same sums up to the order of summation
(double-float and FP64: a tolerance of 1e-11 of the summed magnitudes is thousands of times their rounding), the same
sign-failure counts, and the sums of a subset of sectors must be those of the whole pass."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1508_02512_gb300 import _native as N  # noqa: E402
from paper_1508_02512_gb300 import api  # noqa: E402
from paper_1508_02512_gb300 import tables as T  # noqa: E402


@pytest.fixture(scope="module")
def dbox():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = W.CONFIG3
    blob = T.compile_integral(cfg.topology, T.zero_invariants_of(cfg.topology, cfg.point))
    prep = api.prepare(blob, cfg.kin, cfg.order_min, cfg.order_max)
    return prep, api.DeviceIntegral(prep)


def sums_of(dbox, n, m, block, points, active=None, lam=0.3):
    prep, dev = dbox
    z = [pow(76, j, n) or 1 for j in range(6)]
    p = api.make_pass(n, z, m, 3, N.QMC_PREC_MIXED, block=block, points_per_thread=points)
    if active is not None:
        act = np.ascontiguousarray(active, dtype=np.int32)
        p.sector_active = act.ctypes.data
    sh = torch.tensor(W.shifts(5, m), device="cuda")
    lams = torch.full((prep.info.n_sectors,), lam, dtype=torch.float64, device="cuda")
    sums, fails = dev.outputs(p)
    dev.eval_sums(p, sh, lams, sums, fails)
    torch.cuda.synchronize()
    return sums.cpu().numpy(), fails.cpu().numpy()


# groups per block: 16, 8, 5 (32 threads left over), 4; one point, odd counts, more points than a pair of pairs; lattices
# smaller than an item, one point longer than one, and with a last set that is not full
@pytest.mark.parametrize("n,m,block,points", [(37, 1, 32, 1), (129, 3, 96, 3), (257, 3, 128, 2), (1021, 5, 64, 5),
                                              (2049, 1, 128, 16), (2049, 2, 96, 64)])
def test_sums_do_not_depend_on_the_launch_shape(dbox, n, m, block, points):
    a, fa = sums_of(dbox, n, m, block, points)
    b, fb = sums_of(dbox, n, m, 0, 0)
    assert np.isfinite(a).all()
    scale = np.abs(b).max(axis=(1, 2, 3), keepdims=True)
    assert (np.abs(a - b) <= 1e-11 * scale).all()
    assert np.array_equal(fa, fb)


def test_subset_of_sectors(dbox):
    ns = dbox[0].info.n_sectors
    active = (np.arange(ns) % 3 == 1).astype(np.int32)
    whole, fw = sums_of(dbox, 521, 3, 0, 16)
    part, fp = sums_of(dbox, 521, 3, 0, 16, active)
    on = active != 0
    assert np.array_equal(part[on], whole[on]) and np.array_equal(fp[on], fw[on])
    assert not part[~on].any()
