"""Merging by groups against the oracle: groups of every size class and around their limits, more
HSPs than any group holds, many queries with few HSPs, and runs whose records share query starts."""
import numpy as np
import pytest

import synth
from tests.test_gpu_device_counts import check
from tests.test_gpu_parity import gn  # noqa: F401

pytestmark = pytest.mark.gpu

ALPHABET = np.frombuffer(b"ACGT", dtype=np.uint8)


def bases(rng, n):
    return ALPHABET[rng.integers(0, 4, n)].tobytes()


@pytest.mark.parametrize("top", [0, 1, 100, 1024])
@pytest.mark.parametrize("most", [1500, 8192, 8193])
def test_copies_in_one_sequence(gn, most, top):  # noqa: F811
    """One sequence: a query's HSPs can not be shared out, so its group is as large as its copies."""
    rng = np.random.default_rng(most)
    cores = [bases(rng, 40) for _ in range(8)]
    copies = [most, 1025, 1024, 65, 64, 33, 1, 0]
    if top == 0:  # every alignment is read back: fewer of them
        copies[0] = 8193 if most == 8193 else 1500
    at = rng.permutation(np.repeat(np.arange(8), copies))
    seq = b"".join(cores[i] + bases(rng, int(rng.integers(0, 9))) for i in at)
    qs = synth.queries_from_strings([bases(rng, 7) + c + bases(rng, 5) for c in cores])
    check(gn, synth.bank_from_strings([seq]), qs, stride=4, max_alignments=top, band_w=4)


@pytest.mark.parametrize("top", [0, 2, 100])
def test_shared_starts_and_long_runs(gn, top):  # noqa: F811
    """Repeats in bank and queries: many HSPs of one query start, boxes that grow over several
    records, and sequences whose records overlap from end to end, over many groups."""
    rng = np.random.default_rng(5)
    unit, core = bases(rng, 48), bases(rng, 300)
    seqs = []
    for i in range(400):
        c = bytearray(core)
        for p in rng.integers(0, 300, int(rng.integers(0, 25))):
            c[p] = int(rng.choice(ALPHABET))
        if i % 2:
            del c[150:150 + int(rng.integers(1, 9))]
        seqs.append(bases(rng, int(rng.integers(0, 60))) + bytes(c) + unit * int(rng.integers(0, 4)))
    queries = [unit * 3 + core + unit, core[:170], unit * 2, core[100:] + bases(rng, 30) + core[:120], bases(rng, 99)]
    check(gn, synth.bank_from_strings(seqs), synth.queries_from_strings(queries), stride=4, max_alignments=top, band_w=5)


@pytest.mark.parametrize("top", [0, 100])
def test_short_query_of_a_frequent_repeat(gn, top):  # noqa: F811
    """Most HSPs belong to one short query: its groups follow from its HSPs, not from its length."""
    rng = np.random.default_rng(8)
    core, other = bases(rng, 44), bases(rng, 30_000)
    seqs = [core[:int(rng.integers(30, 45))] + bases(rng, int(rng.integers(0, 9))) for _ in range(9000)]
    seqs += [other[500 * i:500 * i + 300] for i in range(60)]
    check(gn, synth.bank_from_strings(seqs), synth.queries_from_strings([other, core, other[::-1]]), stride=4, max_alignments=top,
          band_w=4, max_evalue=1e-3 if top == 0 else float("inf"))


def test_many_queries(gn):  # noqa: F811
    """More queries than the merge in one block takes, most with one HSP or none."""
    rng = np.random.default_rng(6)
    src = [bases(rng, 90) for _ in range(300)]
    queries = [src[int(rng.integers(300))][:int(rng.integers(30, 90))] if i % 3 else bases(rng, 25) for i in range(4100)]
    check(gn, synth.bank_from_strings(src), synth.queries_from_strings(queries), max_alignments=3)


@pytest.mark.parametrize("top", [0, 100])
@pytest.mark.parametrize("copies", [40, 1500, 9000])
def test_join_of_long_queries(gn, copies, top):  # noqa: F811
    """Pieces of a query in segments: chains that cross segments, and in one sequence as many short
    ones as no group holds."""
    rng = np.random.default_rng(copies)
    q = bases(rng, 140_000)
    many = b"".join(q[a:a + 36] + bases(rng, int(rng.integers(0, 5))) for a in rng.integers(0, 139_000, copies))
    far = bytearray(q[30_000:139_900])
    for p in rng.integers(0, len(far), 300):
        far[p] = int(rng.choice(ALPHABET))
    seqs = [many, bytes(far), q[56_000:66_000], bases(rng, 500), q[57_000:57_400] + q[:300], q[100:400]]
    check(gn, synth.bank_from_strings(seqs), synth.queries_from_strings([q, q[1000:1500], b"", q[65_000:139_000]]), stride=4,
          max_alignments=top, band_w=4, max_evalue=1e-3 if top == 0 else float("inf"))
