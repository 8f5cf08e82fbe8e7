"""Small calls against the oracle: list units summed by the last block around the sizes of warps,
blocks and its limit, and boxes whose band only the wide kernel or the strips hold."""
import numpy as np
import pytest

import synth
from tests.test_gpu_device_counts import check
from tests.test_gpu_parity import gn  # noqa: F401

pytestmark = pytest.mark.gpu

ALPHABET = np.frombuffer(b"ACGT", dtype=np.uint8)


def bases(rng, n):
    return ALPHABET[rng.integers(0, 4, n)].tobytes()


@pytest.mark.parametrize("stride", [11, 1])
@pytest.mark.parametrize("total", [40, 255, 256, 257, 4095, 4096, 4097, 4400])
def test_query_offsets(gn, total, stride):  # noqa: F811
    rng = np.random.default_rng(total)
    src = [bases(rng, 1500) for _ in range(6)]
    queries, left = [], total
    while left:
        n = min(left, int(rng.integers(30, 900)) if left > 60 else left)
        a = int(rng.integers(0, 1500 - n))
        queries.append(src[int(rng.integers(6))][a:a + n])
        left -= n
    assert sum(map(len, queries)) == total
    check(gn, synth.bank_from_strings(src + [src[0][:700]]), synth.queries_from_strings(queries), stride=stride, band_w=5)


@pytest.mark.parametrize("unit", [70, 300])
@pytest.mark.parametrize("n", [1, 5])
def test_wide_boxes(gn, unit, n):  # noqa: F811
    """Tandem copies: overlapping boxes of diagonals a unit apart become one whose band is far wider
    than the default's, beside alignments of the default band."""
    rng = np.random.default_rng(unit + n)
    u, other = bases(rng, unit), bases(rng, 400)
    seqs = [bases(rng, 50) + u * 3 + bases(rng, 20), other, bases(rng, 300)]
    queries = [u * 2 + u[:unit // 2] for _ in range(n)] + [other[20:350]]
    check(gn, synth.bank_from_strings(seqs), synth.queries_from_strings(queries))
