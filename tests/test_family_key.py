"""The generated code of an image is looked up by what the image holds, not by the family its header names: an image whose
terms differ from those that the header's family was taken from (edited, or put together by another program) gets its own
code.  Checked without a device through the disk cache of compiled modules."""
import ctypes
import os

import numpy as np

import workloads as W
from paper_1508_02512_gb300 import api
from paper_1508_02512_gb300 import tables as T
from test_generated_source import PackedHeader, image


def prepared(swap=False):
    """the massive box; swap: with the first two variables of every sector exchanged, which keeps all sizes"""
    cfg = W.CONFIG1
    meta, leaves = T.read_table(T.compile_integral(cfg.topology, T.zero_invariants_of(cfg.topology, cfg.point)))
    if swap:
        order = [1, 0, 2]
        for s in leaves:
            s.A, s.B = s.A[order], s.B[order]
            s.U, s.F = T.Poly(s.U.e[:, order], s.U.c), T.Poly(s.F.e[:, order], s.F.c)
    return api.prepare(T.write_table(leaves, meta), cfg.kin, cfg.order_min, cfg.order_max)


def test_look_up_does_not_rest_on_the_header(tmp_path, monkeypatch):
    monkeypatch.setenv("QMC_GEN_CACHE_DIR", str(tmp_path))
    a, b = prepared(), prepared(swap=True)
    ha, hb = image(a)[0], image(b)[0]
    assert ha.family != hb.family and len(a.packed) == len(b.packed)
    for f in ("dim", "n_sectors", "n_terms_total", "max_terms", "eU0", "eU1", "eF0", "eF1"):
        assert getattr(ha, f) == getattr(hb, f)
    first = api.gen_compile(a, load=False)
    raw = bytearray(b.packed)
    at = PackedHeader.family.offset
    raw[at:at + 8] = bytes(ctypes.c_uint64(ha.family))
    b.packed = bytes(raw)
    assert image(b)[0].family == ha.family
    second = api.gen_compile(b, load=False)
    assert first.cached == 0 and second.cached == 0 and first.family != second.family
    assert len(os.listdir(tmp_path)) == 2


def test_every_exponent_counts():
    """one exponent of one term changed in the packed image, anywhere: another family"""
    prep = prepared()
    h, secs, terms = image(prep)
    rng = np.random.Generator(np.random.PCG64(0))
    seen = {api.gen_compile(prep, load=False).family}
    for term in rng.choice(h.n_terms_total, 4, replace=False):
        raw = bytearray(prep.packed)
        raw[h.termsf_off + 16 * int(term) + 8 + int(rng.integers(0, 3))] ^= 4
        seen.add(api.gen_compile(api.Prepared(bytes(raw), None), load=False).family)
    assert len(seen) == 5
