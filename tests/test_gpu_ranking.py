"""Ranking in registers against the oracle: around the sizes of its teams, equal scores within and
across sequences, repeated ranges, and sequence numbers of more bits than a key holds."""
import os

import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_device_counts import check
from tests.test_gpu_parity import assert_ranked_equal, gn  # noqa: F401

pytestmark = pytest.mark.gpu

ALPHABET = np.frombuffer(b"ACGT", dtype=np.uint8)


@pytest.mark.parametrize("top", [31, 32, 127, 128, 129, 257, 1023, 1024])
def test_team_limits(gn, top):  # noqa: F811
    """One sequence and many: a query's alignments, up to `top`, with few distinct scores, and tandem
    copies whose wide bands find one alignment several times."""
    rng = np.random.default_rng(top)
    core, unit = ALPHABET[rng.integers(0, 4, 48)].tobytes(), ALPHABET[rng.integers(0, 4, 30)].tobytes()
    pieces = []
    for i in range(1100):
        c = bytearray(core[:int(rng.integers(40, 49))])
        if i % 4 == 0:
            c[int(rng.integers(30, 40))] = int(rng.choice(ALPHABET))
        pieces.append(bytes(c) + ALPHABET[rng.integers(0, 4, int(rng.integers(0, 7)))].tobytes())
    seqs = [b"".join(pieces[:700])] + pieces[700:] + [unit * 6 + unit[:11] + unit * 5 for _ in range(9)]
    qs = synth.queries_from_strings([core, core[:44] + unit * 4, unit * 3, core[::-1]])
    check(gn, synth.bank_from_strings(seqs), qs, stride=4, max_alignments=top, band_w=24)


@pytest.mark.parametrize("top", [100, 200])
def test_sequence_numbers_of_24_bits(gn, top):  # noqa: F811
    rng = np.random.default_rng(4)
    n = (1 << 23) + 301
    bases = ALPHABET[rng.integers(0, 4, n * 24, dtype=np.uint8)]
    core = ALPHABET[rng.integers(0, 4, 24)]
    at = np.concatenate([np.arange(a, a + 24) for a in (0, 1001, 1 << 22, (1 << 23) - 9, n - 24)])
    for i in at:
        seq = core.copy()
        if rng.random() < 0.4:
            seq[int(rng.integers(22, 24))] = ALPHABET[int(rng.integers(4))]
        bases[24 * i:24 * i + 24] = seq
    bank = synth.Bank(np.arange(n + 1, dtype=np.uint64) * np.uint64(24), bases, synth.BANKS["tiny"])
    qs = synth.queries_from_strings([core.tobytes(), core[1:].tobytes()])
    ix = gn.Index.from_bank(bank)
    res = gn.search(ix, qs.start, qs.bases, params=gn.make_params(max_alignments=top))
    ref = oracle.Index(bank, restrict_to=qs, threads=os.cpu_count() or 1).search(qs, oracle.Params(max_alignments=top), threads=2)
    assert len(ref[0].ranked) == min(top, 120)
    for i in range(qs.n):
        assert_ranked_equal(res.query(i), ref[i].ranked, f"query {i}")
    ix.close()
