"""Spaced seeds whose mask begins or ends with positions that are not kept: a window is a hit only
where all of it lies in the query and in the sequence, not its kept positions alone.  Every phase
of the signature scan against the oracle, with copies that end 0 to a span of bases before the
ends of queries and sequences."""
import os

import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_parity import check_stages, gn  # noqa: F401

pytestmark = pytest.mark.gpu


def case(span, seed):
    rng = np.random.default_rng(seed)
    alphabet = np.frombuffer(b"ACGT", dtype=np.uint8)
    rand = lambda n: alphabet[rng.integers(0, 4, n)].tobytes()
    src = rand(3000)
    seqs, queries = [], []
    for cut in range(span + 1):  # a copy with `cut` other bases after it, or before it, at the sequence's end
        a, n = int(rng.integers(0, 2000)), int(rng.integers(2 * span, 400))
        seqs += [src[a:a + n] + rand(cut), rand(cut) + src[a:a + n], src[a:a + n]]
        queries += [src[a:a + n + cut], src[max(0, a - cut):a + n], src[a:a + n] + rand(cut), rand(cut) + src[a:a + n]]
    seqs += [src, src[:2000] + rand(1)]  # chains longer than a lane's walk
    queries += [src, src[3:] + rand(2), src[:span], src[:span + 1]]
    return synth.bank_from_strings(seqs), synth.queries_from_strings(queries)


# at strides 29 and 40 the windows in reach of a hit span more than 64 bases
@pytest.mark.parametrize("t", [7, 3, 29, 40])
@pytest.mark.parametrize("mask", ["1101100", "0011011", "0110110", "0011110", "00011011000"])
def test_windows_that_hang_over_an_end_are_no_hits(gn, mask, t):  # noqa: F811
    bank, qs = case(len(mask), 10 * t + len(mask))
    k = mask.count("1")
    p = dict(min_hsp_len=len(mask) + 1, band_w=4)
    ix = gn.Index.from_bank(bank, k=k, stride=t, mask=mask)
    res = gn.search(ix, qs.start, qs.bases, params=gn.make_params(flags=gn.GN_FLAG_KEEP_STAGES, **p))
    ref = oracle.Index(bank, k=k, stride=t, mask=mask).search(qs, oracle.Params(k=k, stride=t, **p),
                                                              threads=os.cpu_count() or 1)
    assert sum(len(r.hsp) for r in ref) > 0
    check_stages(gn, res, ref, qs.n, f"mask {mask} stride {t}")
    ix.close()
