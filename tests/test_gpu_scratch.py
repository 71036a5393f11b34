"""What a call may need: a setup whose tables fill the shared memory of the per-segment FFT fit."""
import numpy as np
import pytest

import synth
from oracle import reference as R
from tests.gpu_helpers import assert_fit_match
from tests.test_gpu_tree import frbx, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


def test_setup_that_fills_shared_memory(frbx):  # noqa: F811
    """38 channels x 128 points on a grid of 512 x 2048: 232112 bytes of tables and 336 of the kernel's own are all that
    a CTA can have."""
    g = np.r_[0:37, 1023]
    wl = synth.make_tiny(n_chan=38, n_point=128, T=20, n_bl=2, dms=(0.0, 5.0), windows=[3], f0=3000.0 + 16.0 * g, pulse=False)
    wl.sbd_pad = 4
    st = R.setup_from_workload(wl)
    assert (st.Ls, st.Lm) == (512, 2048)
    vis = synth.generate(wl)
    dk = R.shift_table(st, wl.dms)
    segs, idx, _ = R.all_segments(20, 2, [3], dk.max(axis=1))
    segs, idx = segs[:6], idx[:6]
    ref = R.fit_segments(st, vis, dk, segs)
    h = frbx.Handle.from_workload(wl)
    assert_fit_match(st, vis, dk, segs, h.fit_segments(to_dev(vis), wl.dms, segs, kernel=2), ref)
    ser = h.search(to_dev(vis), wl.dms, [3], want_series=True)["series"]
    assert_fit_match(st, vis, dk, segs, ser.reshape(-1)[idx], ref)
