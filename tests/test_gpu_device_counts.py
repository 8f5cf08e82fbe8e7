"""Searches whose counts stay on the device, against the oracle: merging in one block and over the
whole call around its limit, queries with more alignments than a block ranks, selection by
lengths of three bytes, equally long boxes, alignment orders around their limits, and bands that
only the strip path holds."""
import os

import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_parity import assert_ranked_equal, gn  # noqa: F401

pytestmark = pytest.mark.gpu

ALPHABET = np.frombuffer(b"ACGT", dtype=np.uint8)


def check(g, bank, qs, stride=11, **kw):
    ix = g.Index.from_bank(bank, stride=stride)
    res = g.search(ix, qs.start, qs.bases, params=g.make_params(**kw))
    ref = oracle.Index(bank, stride=stride).search(qs, oracle.Params(stride=stride, **kw), threads=os.cpu_count() or 1)
    assert sum(len(r.ranked) for r in ref) > 0
    for i in range(qs.n):
        assert_ranked_equal(res.query(i), ref[i].ranked, f"query {i} {kw}")
    whole = res.all()
    assert len(whole) == qs.n and all(np.array_equal(a, res.query(i)) for i, a in enumerate(whole))
    ix.close()


@pytest.mark.parametrize("top", [0, 3, 100, 1024, 1025])
@pytest.mark.parametrize("n", [1, 33, 513, 970, 1000, 1025, 2049])
def test_many_copies(gn, n, top):  # noqa: F811
    """n sequences with one diverged copy each of a query's middle: n HSPs, or nearly."""
    rng = np.random.default_rng(n)
    rand = lambda k: ALPHABET[rng.integers(0, 4, k)].tobytes()
    core = rand(70)
    seqs = []
    for i in range(n):
        c = bytearray(core)
        if i % 3:
            c[int(rng.integers(40, 70))] = int(rng.choice(ALPHABET))
        seqs.append(rand(int(rng.integers(0, 30))) + bytes(c) + rand(int(rng.integers(0, 12))))
    qs = synth.queries_from_strings([rand(13) + core + rand(9), rand(40), core[:44], b""])
    check(gn, synth.bank_from_strings(seqs), qs, stride=4, max_alignments=top, band_w=6,
          max_evalue=1e-3 if n == 513 else float("inf"))


@pytest.mark.parametrize("top", [1, 2, 5])
@pytest.mark.parametrize("stride", [11, 1])
def test_equally_long_boxes(gn, stride, top):  # noqa: F811
    """Tandem repeats: many boxes of one length per query, cut after the first few in (sequence,
    query start, bank start) order."""
    rng = np.random.default_rng(3 + stride)
    rand = lambda k: ALPHABET[rng.integers(0, 4, k)].tobytes()
    unit = rand(66)
    seqs = []
    for _ in range(50):
        body = bytearray(unit * int(rng.integers(2, 7)))
        for _ in range(int(rng.integers(0, 4))):
            body[int(rng.integers(len(body)))] = int(rng.choice(ALPHABET))
        seqs.append(rand(int(rng.integers(0, 99))) + bytes(body) + rand(int(rng.integers(0, 99))))
    queries = [rand(int(rng.integers(0, 30))) + unit * int(rng.integers(1, 5)) + unit[:int(rng.integers(0, 66))]
               for _ in range(14)]
    check(gn, synth.bank_from_strings(seqs), synth.queries_from_strings(queries), stride=stride, max_alignments=top)


@pytest.mark.parametrize("top", [1, 3, 100])
def test_selection_of_lengths_over_16_bits(gn, top):  # noqa: F811
    rng = np.random.default_rng(9)
    rand = lambda k: ALPHABET[rng.integers(0, 4, k)].tobytes()
    q = rand(140_000)
    seqs = [q[:66_000], q[1000:67_000], q[70_000:70_300], q[80_000:80_290] + rand(50), q[2:65_538], q[90_000:90_256],
            q[100_000:100_255], rand(500)]
    check(gn, synth.bank_from_strings(seqs), synth.queries_from_strings([q, q[:400]]), max_alignments=top)


@pytest.mark.parametrize("w", [16, 60, 150, 700])
@pytest.mark.parametrize("nq", [3, 700])
def test_alignment_order_and_strips(gn, nq, w):  # noqa: F811
    """Few and many alignments, of lengths over several factors of two, on every band path."""
    rng = np.random.default_rng(nq)
    rand = lambda k: ALPHABET[rng.integers(0, 4, k)].tobytes()
    src = [rand(int(k)) for k in np.exp(rng.uniform(np.log(30), np.log(1500), 40))]
    queries = []
    for _ in range(nq):
        c = bytearray(src[int(rng.integers(40))])
        for p in rng.integers(0, len(c), len(c) // 20):
            c[p] = int(rng.choice(ALPHABET))
        if len(c) > 200:
            del c[100:100 + int(rng.integers(0, 25))]
        queries.append(bytes(c) if nq == 3 or len(c) < 400 else bytes(c[:int(rng.integers(60, 400))]))
    check(gn, synth.bank_from_strings(src), synth.queries_from_strings(queries), band_w=w)
