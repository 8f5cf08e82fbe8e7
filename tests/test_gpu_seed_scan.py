"""The signature scan (seed lookup and chaining without storing hits) against the oracle, every
phase, and against the hit-storing bucket path: chains of every link length up to the limit and
one past it, chains longer than a lane's walk, at sequence starts and ends, next to non-bases and
the ends of the bank, lists longer than a tile, windows wider than 64 bases, spaced seeds."""
import os

import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_parity import assert_ranked_equal, check_stages, gn  # noqa: F401

pytestmark = pytest.mark.gpu


def scan_case(seed):
    rng = np.random.default_rng(seed)
    alphabet = np.frombuffer(b"ACGT", dtype=np.uint8)
    rand = lambda n: alphabet[rng.integers(0, 4, n)].tobytes()
    src = rand(6000)
    seqs, queries = [], []
    for i in range(120):  # pieces of one source with changes at set distances, back to back
        a = int(rng.integers(0, 4000))
        s = bytearray(src[a:a + int(rng.integers(1, 1600))])
        for p in range(int(rng.integers(0, 60)), len(s), int(rng.choice([13, 23, 34, 45, 56, 90, 500]))):
            s[p] = int(rng.choice(alphabet)) if i % 3 else ord("N")
        seqs.append(bytes(s))
    seqs += [b"", b"A" * 5000 + src[700:760], rand(7), b"AC" * 150, src, rand(300)]
    seqs.append(src[-40:])  # ends the bank
    for a, n in ((0, 6000), (100, 64), (3000, 2500), (5960, 40), (17, 333)):
        q = bytearray(src[a:a + n])
        queries.append(bytes(q))
        for p in range(9, n, 71):
            q[p] = int(rng.choice(alphabet)) if n != 2500 else ord("n")
        queries.append(bytes(q))
    queries += [b"A" * 13 + src[700:760], b"AC" * 40, b"", rand(10), rand(500), b"N" * 30, src[:22]]
    return synth.bank_from_strings(seqs), synth.queries_from_strings(queries)


# k, stride, mask, hit distance (0: default), minimum length (0: default): both sides of each
# limit of the scan
CASES = [(11, 11, None, 0, 0), (11, 11, None, 11, 0), (11, 11, None, 32, 23), (11, 11, None, 43, 60),
         (11, 11, None, 44, 0), (11, 1, None, 0, 0), (11, 1, None, 1, 16), (11, 1, None, 11, 26), (11, 1, None, 2, 70),
         (11, 1, None, 12, 0), (9, 2, None, 0, 0), (8, 4, None, 9, 0), (11, 30, None, 0, 0), (12, 40, None, 41, 0),
         (13, 13, None, 0, 0), (6, 3, None, 0, 0), (11, 1, "110011011", 0, 0),
         (11, 18, "111010010100110111", 0, 0), (11, 9, "111010010100110111", 0, 24), (11, 40, "1101" + "0" * 24 + "1111", 0, 33)]


@pytest.mark.parametrize("k,t,mask,dist,min_len", CASES)
def test_scan_equals_oracle_and_bucket_path(gn, k, t, mask, dist, min_len, monkeypatch):  # noqa: F811
    bank, qs = scan_case(k * 100 + t)
    kk = mask.count("1") if mask else k
    ix = gn.Index.from_bank(bank, k=k, stride=t, mask=mask)
    ox = oracle.Index(bank, k=kk, stride=t, mask=mask)
    p = dict(max_hit_distance=dist, min_hsp_len=min_len, band_w=8)
    params = gn.make_params(flags=gn.GN_FLAG_KEEP_STAGES, **p)
    res = gn.search(ix, qs.start, qs.bases, params=params)
    ref = ox.search(qs, oracle.Params(k=kk, stride=t, **p), threads=os.cpu_count() or 1)
    check_stages(gn, res, ref, qs.n, f"k {k} stride {t} mask {mask} D {dist} min {min_len}")
    monkeypatch.setenv("GN_HIT_GROUPING", "bucket")
    other = gn.search(ix, qs.start, qs.bases, params=params)
    order = lambda h: np.sort(h, order=list(h.dtype.names))
    assert np.array_equal(order(res.stage(gn.GN_STAGE_HSP)), order(other.stage(gn.GN_STAGE_HSP)))
    ix.close()


@pytest.mark.parametrize("shift", [0, 1, 2, 3, 4, 8, 13])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 63, 64, 65, 700])
def test_packing_of_device_queries_at_any_byte(gn, shift, n):  # noqa: F811
    """Queries that start at any byte of a buffer and end at any offset of a packed word, with
    other letters right before and after them."""
    import torch
    rng = np.random.default_rng(n)
    bank = synth.make_bank("tiny", n_seqs=60)
    ix = gn.Index.from_bank(bank)
    q = bank.bases[500:500 + n].copy()
    q[rng.integers(0, n, n // 40)] = ord("x")
    buf = np.full(n + 64, ord("C"), np.uint8)
    buf[shift:shift + n] = q
    start = np.array([0, n], np.uint64)
    p = gn.make_params(min_hsp_len=11)
    want = gn.search(ix, start, q, params=p).query(0)
    got = gn.search(ix, start, torch.from_numpy(buf).cuda()[shift:shift + n], params=p).query(0)
    assert_ranked_equal(got, oracle.Index(bank).search(synth.queries_from_strings([q.tobytes()]),
                                                       oracle.Params(min_hsp_len=11))[0].ranked)
    assert np.array_equal(got, want)
