"""The signature scan in several ranges of its list units, and with a candidate list that room runs
out for: the same HSPs and hits as the oracle, whatever the ranges cut through (a list, a query, a
chain), and the number of launches that the cut asks for."""
import os

import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_parity import assert_ranked_equal, check_stages, gn  # noqa: F401
from tests.test_gpu_seed_scan import scan_case

pytestmark = pytest.mark.gpu


def check(gn, bank, qs, stride, least, most, ctx):  # noqa: F811
    ix = gn.Index.from_bank(bank, stride=stride)
    res = gn.search(ix, qs.start, qs.bases, params=gn.make_params(flags=gn.GN_FLAG_KEEP_STAGES | gn.GN_FLAG_TIME_KERNELS))
    launches = ix.kernel_times()["k_seed_scan"][1]
    ref = oracle.Index(bank, stride=stride).search(qs, oracle.Params(stride=stride), threads=os.cpu_count() or 1)
    check_stages(gn, res, ref, qs.n, ctx)
    hits = sum(r.n_hits for r in ref)
    assert least(hits) <= launches <= most(hits), (launches, hits)
    ix.close()


@pytest.mark.parametrize("hits", [40, 1000, 4096, 100_000_000])
@pytest.mark.parametrize("stride", [11, 1])
def test_ranges_of_units(gn, stride, hits, monkeypatch):  # noqa: F811
    """Units hold up to four hits, and every offset one at least; a launch is repeated where the first
    list, of 16,384 candidates, is too short."""
    bank, qs = scan_case(5 + stride)
    offsets = int(qs.start[-1])
    monkeypatch.setenv("GN_MAX_CHUNK_HITS", str(hits))
    check(gn, bank, qs, stride, lambda n: offsets // hits or 1, lambda n: 4 * (n + 2 * offsets) // hits + 1 + n // 16384,
          f"stride {stride}, {hits} hits a range")


@pytest.mark.parametrize("room", [4, 33, 1000])
@pytest.mark.parametrize("stride", [11, 1])
def test_room_for_candidates(gn, stride, room, monkeypatch):  # noqa: F811
    """Low-complexity sequence, where every hit is a candidate."""
    bank = synth.bank_from_strings([b"A" * 900 + b"C" * 40, b"AC" * 200 + b"ACGTTGCA" * 30, b"G" * 3, b"ACGTTGCA" * 25])
    qs = synth.queries_from_strings([b"A" * 60, b"ACGTTGCA" * 9, b"T" + b"AC" * 30 + b"GG", b"C" * 45])
    monkeypatch.setenv("GN_CAND_ROOM", str(room))
    check(gn, bank, qs, stride, lambda n: 2, lambda n: 4 * (n + 2 * int(qs.start[-1])) + 64, f"stride {stride}, room {room}")


def test_long_queries_at_stride_one(gn, monkeypatch):  # noqa: F811
    """Runs of equal bases across the ends of segments, whole and a base short of them, in one
    launch and in several."""
    rng = np.random.default_rng(11)
    rand = lambda n: np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, n)].tobytes()
    step, ends = 65535 - 8192, 65535
    q = bytearray(rand(200_000))
    seqs = [rand(300)]
    for at, n in ((step - 40, 80), (ends - 30, 60), (ends - 26, 26), (step, 30), (step + ends - 23, 24), (2 * step - 1, 9000),
                  (ends - 11, 50), (199_950, 50)):
        seqs.append(rand(int(rng.integers(0, 20))) + bytes(q[at:at + n]) + rand(int(rng.integers(0, 20))))
    q[500] = ord("N")
    bank, qs = synth.bank_from_strings(seqs), synth.queries_from_strings([bytes(q), bytes(q[ends - 100:ends + 100]), bytes(q[:ends + 1])])
    ix = gn.Index.from_bank(bank, stride=1)
    ref = oracle.Index(bank, stride=1).search(qs, oracle.Params(stride=1), threads=os.cpu_count() or 1)
    for chunk in (0, 20_000):
        if chunk:
            monkeypatch.setenv("GN_MAX_CHUNK_HITS", str(chunk))
        res = gn.search(ix, qs.start, qs.bases)
        for i in range(qs.n):
            assert_ranked_equal(res.query(i), ref[i].ranked, f"chunk {chunk} query {i}")
        assert len(res.query(0)) >= 8
    ix.close()
