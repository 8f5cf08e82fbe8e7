"""The request loop with one thread that submits and another that collects."""
import threading
import time

import numpy as np
import pytest

import synth
from tests.test_gpu_parity import gn  # noqa: F401

pytestmark = pytest.mark.gpu


def submit_all(gn, ix, requests, collect):  # noqa: F811
    """(seconds that the submissions took, hits of each request)."""
    srv = gn.Server(ix, 4 << 30)
    held = {}

    def collector():
        while len(held) < len(requests):
            got = srv.poll_any(200)
            if got is not None:
                held[got[0]] = got[1]

    th = threading.Thread(target=collector)
    if collect:
        th.start()
    t = time.perf_counter()
    tickets = [srv.submit(r) for r in requests]
    t = time.perf_counter() - t
    if not collect:
        th.start()
    th.join(120)
    out = [held[k].query(0) for k in tickets]
    srv.stop()
    return t, out


def test_collecting_beside_submitting(gn):  # noqa: F811
    """Submitting takes at most three times as long beside a thread that collects as without it: the
    two share one interpreter, which makes it twice as long, and hand it over less than once a request
    (with a hand-over for each poll 3.4 to 3.6 times as long).  Best of eight runs each."""
    bank = synth.make_bank("mid", n_seqs=3000)
    qs = synth.make_queries("mid", bank, n=50)
    requests = [qs.query(i)[:400] for i in range(qs.n)] * 60
    ix = gn.Index.from_bank(bank)
    runs = [(submit_all(gn, ix, requests, False), submit_all(gn, ix, requests, True)) for _ in range(8)]
    alone, beside = (min(r[i][0] for r in runs) for i in (0, 1))
    for a, b in runs:
        for i in range(len(requests)):
            assert np.array_equal(a[1][i], a[1][i % qs.n]) and np.array_equal(b[1][i], a[1][i % qs.n])
    print(f"submitting {1e3 * alone:.1f} ms alone, {1e3 * beside:.1f} ms beside the collector")
    assert beside <= 3 * alone, (alone, beside)
    ix.close()
