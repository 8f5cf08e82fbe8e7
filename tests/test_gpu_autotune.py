"""What the autotuner times: settings that only the hit-storing route has are left at their defaults
where the sample's search does not take it."""
import numpy as np
import pytest

import synth
from tests.test_gpu_parity import gn  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stored", [False, True])
def test_settings_of_the_route_that_the_sample_takes(gn, stored, monkeypatch):  # noqa: F811
    """27 searches with signatures (9 settings of the alignment, three runs each), 54 with stored
    hits (9 more); the installed settings do not change the hits."""
    bank = synth.make_bank("mid", n_seqs=5000)
    qs = synth.make_queries("mid", bank, n=40)
    if stored:
        monkeypatch.setenv("GN_HIT_GROUPING", "bucket")
    ix = gn.Index.from_bank(bank)
    want = gn.search(ix, qs.start, qs.bases).all()
    a = gn.gn_kernel_launch_count()
    gn.search(ix, qs.start, qs.bases)
    b = gn.gn_kernel_launch_count()
    _, t = gn.autotune(ix, qs.start, qs.bases, what=gn.GN_TUNE_KERNELS)
    c = gn.gn_kernel_launch_count()
    searches = (c - b) / (b - a)  # settings may add a launch or two to a search's nine or more
    if stored:
        assert searches > 40
        assert t["fill_threads"] in (256, 512) and t["tile_hits"] in (25000, 50000, 100000) and t["bucket_target"] in (2048, 4096, 8192)
    else:
        assert searches < 33
        assert (t["fill_threads"], t["tile_hits"], t["bucket_target"]) == (512, 50000, 4096)
    got = gn.search(ix, qs.start, qs.bases).all()
    assert all(np.array_equal(x, y) for x, y in zip(got, want))
    ix.close()
