"""What a batch object keeps between calls: the captured graph when the DM trials that leave an AP change."""
import numpy as np
import pytest

import synth
from tests.test_gpu_batch import _same
from tests.test_gpu_tree import frbx, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [synth.make_vgos, synth.make_small])
def test_more_trials_that_leave_an_ap(frbx, make):  # noqa: F811
    """Two DM lists of one length; sweeps of the first one's last trials are longer than the scans."""
    kw = {"n_dm": 6} if make is synth.make_vgos else {}
    wls = [make(T=T, n_bl=2, seed_offset=0, **kw) for T in (300, 260)]
    for wl in wls:
        wl.pulses = []
    h = frbx.Handle.from_workload(wls[0])
    h.set_limits(tree_chunk_bytes=1 << 20)
    vis = [to_dev(synth.generate(wl)) for wl in wls]
    lists = [np.array([0.0, 1.0, 2.0, 9e4, 9e4, 9e4]), np.array([0.0, 1.0, 2.0, 3.0, 4.0, 5.0]), np.array([0.0, 9e4, 9e4, 9e4, 9e4, 9e4])]
    ref = frbx.Handle.from_workload(wls[0])
    with frbx.Batch() as b:
        for k, dms in enumerate(lists):
            out = b.search([(h, v) for v in vis], dms, [2, 4, 8], want_series=True, want_events=True)
            assert b.info()["graph_captures"] == k + 1
            for v, o in zip(vis, out):
                _same(o, ref.search(v, dms, [2, 4, 8], want_series=True, want_events=True))
        b.search([(h, v) for v in vis], lists[-1], [2, 4, 8])
        assert b.info()["graph_captures"] == len(lists)
