"""X-drop extension: HSPs around the number at which a warp's idle lanes get new walks, walks of less
than a window, a window and many of them in one warp, ends next to the first and last base of the
query and the bank.  HSPs and extensions against the oracle."""
import os

import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_parity import check_stages, gn  # noqa: F401

pytestmark = pytest.mark.gpu

OTHER = bytes.maketrans(b"ACGT", b"CATG")


def stretch(src, step):
    """src with every step-th base another one: no seed of 11, and X-drop goes on through it."""
    b = bytearray(src)
    for i in range(step - 1, len(b), step):
        b[i] = OTHER[b[i]]
    return bytes(b)


@pytest.mark.parametrize("n", [1, 11, 12, 13, 16, 17, 200])
@pytest.mark.parametrize("edge", [0, 5, 31, 32])
def test_walks_of_all_lengths_in_a_warp(gn, n, edge):  # noqa: F811
    rng = np.random.default_rng(100 * n + edge)
    rand = lambda k: np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, k)].tobytes()
    core = rand(33)
    left, right = rand(700), rand(700)
    seqs, lengths = [], [0, 1, 31, 32, 33, 64, 300, 650]
    for i in range(n):
        a, b = int(rng.choice(lengths)), int(rng.choice(lengths))
        # (walked to the left, the changes lie step apart from the core as well)
        seqs.append(rand(int(rng.integers(0, 60))) + stretch(left[700 - a:][::-1], 9)[::-1] + core + stretch(right[:b], 9) +
                    rand(int(rng.integers(0, 60))))
    q = left + core + right
    short = left[700 - edge:] + core + right[:edge]
    # the bank begins and ends with a core that is `edge` bases from its ends
    bank = synth.bank_from_strings([short] + seqs + [short])
    qs = synth.queries_from_strings([q, short, q[200:]])
    ix = gn.Index.from_bank(bank, stride=3)
    res = gn.search(ix, qs.start, qs.bases, params=gn.make_params(flags=gn.GN_FLAG_KEEP_STAGES))
    ref = oracle.Index(bank, stride=3).search(qs, oracle.Params(stride=3), threads=os.cpu_count() or 1)
    check_stages(gn, res, ref, qs.n, f"{n} copies, edge {edge}")
    assert sum(len(r.hsp) for r in ref) >= 3 * n
    ix.close()
