"""Hits do not depend on whether the stage outputs are kept."""
import os

import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_parity import assert_ranked_equal, gn  # noqa: F401

pytestmark = pytest.mark.gpu


def tandem_case(seed, unit_len):
    """Tandem repeats with many changes: boxes of one query start and length, of which a later one
    reaches further back in the sequence than an earlier one."""
    rng = np.random.default_rng(seed)
    alphabet = np.frombuffer(b"ACGT", np.uint8)
    rand = lambda k: alphabet[rng.integers(0, 4, k)].tobytes()
    unit = rand(unit_len)

    def tandem(n):
        b = bytearray(unit * n)
        for _ in range(int(rng.integers(0, 10))):
            b[int(rng.integers(len(b)))] = int(rng.choice(alphabet))
        return bytes(b)

    seqs = [rand(int(rng.integers(0, 30))) + tandem(int(rng.integers(3, 12))) + rand(int(rng.integers(0, 30))) for _ in range(60)]
    queries = [rand(int(rng.integers(0, 20))) + tandem(int(rng.integers(1, 4))) + rand(int(rng.integers(0, 9))) for _ in range(10)]
    return synth.bank_from_strings(seqs), queries


# the query of each case that has such boxes, alone (HSPs merged in one block where they are few) and
# among the others
@pytest.mark.parametrize("seed,unit,k,stride,xdrop,query", [(9, 34, 8, 4, 3, 5), (1, 55, 6, 2, 3, 8), (32, 34, 6, 3, 0, 9)])
@pytest.mark.parametrize("alone", [True, False])
def test_hits_with_and_without_stages(gn, seed, unit, k, stride, xdrop, query, alone):  # noqa: F811
    bank, queries = tandem_case(seed, unit)
    qs = synth.queries_from_strings([queries[query]] if alone else queries)
    ix, ox = gn.Index.from_bank(bank, k=k, stride=stride), oracle.Index(bank, k=k, stride=stride)
    for top in range(1, 26):
        p = dict(max_alignments=top, xdrop=xdrop)
        with_, without = (gn.search(ix, qs.start, qs.bases, params=gn.make_params(flags=f, **p)).all()
                          for f in (gn.GN_FLAG_KEEP_STAGES, 0))
        ref = ox.search(qs, oracle.Params(k=k, stride=stride, **p), threads=os.cpu_count() or 1)
        for i in range(qs.n):
            assert_ranked_equal(without[i], ref[i].ranked, f"top {top} query {i}")
            assert np.array_equal(with_[i], without[i]), (top, i)
    ix.close()
