"""Alignments around the limits of the packed cells (rows, scores, and gap and mismatch scores that
a word holds) against the oracle, on the register bands and the wide ones."""
import os

import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_parity import assert_ranked_equal, gn  # noqa: F401

pytestmark = pytest.mark.gpu

ALPHABET = np.frombuffer(b"ACGT", dtype=np.uint8)
LIMITS = [  # band_w, rows and scores that fit
    (16, 2047, 2047),
    (40, 511, 1023),
]
SCORES = [(1, -3, -5, -2), (4, -5, -2, -2), (7, -9, -3, 0), (1, -511, -400, -111), (1, -512, -5, -2), (1, -3, -400, -112),
          (1, -1023, -1000, -23), (1, -1024, 0, -1), (2, -3, -1000, -24), (1, -2, 0, -1023), (1, -2, 0, -1024)]


@pytest.mark.parametrize("scores", SCORES)
@pytest.mark.parametrize("w,rows,score", LIMITS)
def test_limits(gn, w, rows, score, scores):  # noqa: F811
    rng = np.random.default_rng(rows)
    seqs, queries = [], []
    for limit in sorted({rows, min(rows, score // scores[0])}):
        for n in range(limit - 2 * w - 1, limit - 2 * w + 3):  # copies of n bases: n + 2 w rows
            core = ALPHABET[rng.integers(0, 4, n)].tobytes()
            ends = [ALPHABET[rng.integers(0, 4, 60)].tobytes() for _ in range(4)]
            seqs.append(ends[0] + core + ends[1])
            queries.append(ends[2] + core + ends[3])
            gap = bytearray(core)  # the same with gaps and substitutions, and with a repeat that ties
            del gap[n // 3:n // 3 + 3]
            gap[n // 2] = ord("A") if gap[n // 2] != ord("A") else ord("C")
            gap[2 * n // 3:2 * n // 3] = gap[2 * n // 3 - 6:2 * n // 3]
            seqs.append(ends[1] + bytes(gap) + ends[0])
    bank, qs = synth.bank_from_strings(seqs), synth.queries_from_strings(queries)
    sc = dict(zip(("match", "mismatch", "gap_open", "gap_extend"), scores))
    ix = gn.Index.from_bank(bank)
    res = gn.search(ix, qs.start, qs.bases, scoring=gn.make_scoring(**sc), params=gn.make_params(band_w=w))
    ref = oracle.Index(bank).search(qs, oracle.Params(band_w=w, **sc), threads=os.cpu_count() or 1)
    for i in range(qs.n):
        assert len(ref[i].ranked) > 0
        assert_ranked_equal(res.query(i), ref[i].ranked, f"scores {scores} w {w} query {i}")
    ix.close()
