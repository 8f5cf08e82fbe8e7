"""Device memory that calls hold, by the memory pool's high-water mark."""
import ctypes
import os

import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_parity import assert_ranked_equal, gn  # noqa: F401

pytestmark = pytest.mark.gpu

USED_MEM_HIGH = 8  # CU_MEMPOOL_ATTR_USED_MEM_HIGH


class PoolHigh:
    """Bytes in use of the device's default memory pool, at most, since the last reset()."""

    def __init__(self):
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.pool = ctypes.c_void_p()
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def reset(self):
        assert self.cu.cuMemPoolSetAttribute(self.pool, USED_MEM_HIGH, ctypes.byref(ctypes.c_uint64(0))) == 0

    def value(self):
        v = ctypes.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.pool, USED_MEM_HIGH, ctypes.byref(v)) == 0
        return v.value


def test_all_alignments_of_many_hsps_that_merge(gn):  # noqa: F811
    """Tandem repeats: 1.4 M HSPs of 16,000 boxes.  Room for every alignment is room for the boxes,
    about 170 bytes each: against the call that keeps one a query, no more than that and 16 MiB."""
    rng = np.random.default_rng(2)
    rand = lambda n: np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, n)].tobytes()
    units = [rand(11) for _ in range(5)]
    bank = synth.bank_from_strings([rand(11 * int(rng.integers(0, 3))) + units[i % 5] * 45 + rand(20) for i in range(2000)])
    qs = synth.queries_from_strings([rand(int(rng.integers(0, 20))) + units[i % 5] * 45 + rand(9) for i in range(40)])
    ix = gn.Index.from_bank(bank)
    high = PoolHigh()
    used = {}
    for top in (1, 0):
        gn.search(ix, qs.start, qs.bases, params=gn.make_params(max_alignments=top, band_w=3))
        high.reset()
        res = gn.search(ix, qs.start, qs.bases, params=gn.make_params(max_alignments=top, band_w=3))
        used[top] = high.value()
    ref = oracle.Index(bank).search(qs, oracle.Params(max_alignments=0, band_w=3), threads=os.cpu_count() or 1)
    assert sum(len(r.hsp) for r in ref) > 1 << 20
    boxes = sum(len(r.merged) for r in ref)
    for i in range(qs.n):
        assert_ranked_equal(res.query(i), ref[i].ranked, f"query {i}")
    assert used[0] <= used[1] + 200 * boxes + (16 << 20), (used, boxes)
    ix.close()


def test_signatures_leave_memory_free(gn, monkeypatch, tmp_path):  # noqa: F811
    """An index whose signatures would not leave the reserve free does without them, built or
    loaded: 4 bytes an occurrence less, the same hits."""
    bank = synth.make_bank("mid", n_seqs=2000)
    qs = synth.make_queries("mid", bank, n=20)
    ix = gn.Index.from_bank(bank)
    path = str(tmp_path / "ix.gnx")
    ix.save(path)
    info, want = ix.info(), gn.search(ix, qs.start, qs.bases).all()
    ix.close()
    for reserve, saved in ((1 << 50, 4 * info.n_postings), (0, 0)):
        monkeypatch.setenv("GN_SIGNATURE_RESERVE", str(reserve))
        for make in (lambda: gn.Index.from_bank(bank), lambda: gn.Index.load(path)):
            ix = make()
            assert ix.info().device_bytes == info.device_bytes - saved
            got = gn.search(ix, qs.start, qs.bases).all()
            assert all(np.array_equal(a, b) for a, b in zip(got, want))
            ix.close()
