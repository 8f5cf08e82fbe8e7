"""Banded alignment against the oracle at the widths where its paths meet (a band of one diagonal,
the register paths' 40, 48, 64 and 288 offsets and one more), with alignments a warp each and
grouped, and with scores for which cells past the band have to be cut off (mismatch below twice
the gap extension) and free gaps."""
import os

import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_parity import assert_ranked_equal, gn  # noqa: F401

pytestmark = pytest.mark.gpu

LONG = "GN_SW_LONG_ROWS"
SCORES = [(1, -3, -5, -2), (2, -3, -4, -1), (1, -1, 0, -1), (5, -4, 0, 0), (1, -3, -12, 0), (3, -2, -1, -3)]


@pytest.fixture(scope="module")
def diverged(gn):  # noqa: F811
    rng = np.random.default_rng(77)
    alphabet = np.frombuffer(b"ACGT", dtype=np.uint8)
    rand = lambda n: alphabet[rng.integers(0, 4, n)].tobytes()
    seqs, queries = [], []
    for i in range(60):
        src = rand(int(rng.integers(60, 700)))
        out = bytearray()
        for j, ch in enumerate(src):  # substitutions, runs of inserted and deleted bases, non-bases
            u = rng.random()
            if u < 0.03:
                out += rand(1)
            elif u < 0.045:
                out += bytes([ch]) + rand(int(rng.integers(1, 13)))
            elif u < 0.055:
                continue
            elif u < 0.058:
                out += b"N"
            else:
                out.append(ch)
        cut = int(rng.integers(0, 9))
        if i % 5 == 0:
            del out[len(out) // 2:len(out) // 2 + 11]
        seqs.append(rand(int(rng.integers(0, 40))) + src + rand(int(rng.integers(0, 40))) if i % 4 else src)
        queries.append(bytes(out[cut:]) if i % 3 else rand(20) + bytes(out) + rand(25))
    bank, qs = synth.bank_from_strings(seqs), synth.queries_from_strings(queries)
    return qs, gn.Index.from_bank(bank), oracle.Index(bank)


CASES = [(sc, w, {}) for sc in SCORES for w in (0, 1, 16, 19, 20, 23, 24, 31, 32, 100, 143, 144)]
CASES += [(SCORES[0], w, env) for w in (0, 1, 16, 19, 20, 23, 24)
          for env in ({LONG: "100000"}, {"GN_SW_LANES": "16", LONG: "100000"})]  # grouped: several to a warp
CASES += [(sc, 16, {LONG: "100000"}) for sc in SCORES[1:]]


@pytest.mark.parametrize("scores,w,env", CASES)
def test_bands_equal_oracle(gn, diverged, scores, w, env, monkeypatch):  # noqa: F811
    qs, ix, ox = diverged
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    sc = dict(zip(("match", "mismatch", "gap_open", "gap_extend"), scores))
    res = gn.search(ix, qs.start, qs.bases, scoring=gn.make_scoring(**sc), params=gn.make_params(band_w=w))
    ref = ox.search(qs, oracle.Params(band_w=w, **sc), threads=os.cpu_count() or 1)
    for i in range(qs.n):
        assert_ranked_equal(res.query(i), ref[i].ranked, f"scores {scores} w {w} query {i}")
