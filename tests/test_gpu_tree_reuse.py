"""Many short time tiles of the tensor-core window tree in a row, so that each SM runs several CTAs whose last AP
stores a window anchor to tensor memory just before the columns go to the next CTA.  Every DM trial is the
same (DM 0), so every series has to be the same, and the first one is checked against the FP64 oracle."""
import numpy as np
import pytest

import synth
from oracle import reference as R
from tests.gpu_helpers import assert_fit_match
from tests.test_gpu_tree import frbx, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [2, 4, 6, 10])
@pytest.mark.parametrize("windows", [[4], [1, 2, 4], [64, 2]])
def test_short_tiles_in_a_row(frbx, T, windows):  # noqa: F811
    n_dm = 400  # three column blocks each: about eight CTAs per SM
    wl = synth.make_tiny(n_chan=5, n_point=64, T=T, n_bl=1, dms=np.zeros(n_dm), windows=windows, pulse=False,
                         f0=3000.0 + 16.0 * np.array([0, 3, 33, 50, 63], float))
    st = R.setup_from_workload(wl)
    vis = synth.generate(wl)
    h = frbx.Handle.from_workload(wl)
    ser = h.search(to_dev(vis), wl.dms, windows, want_series=True, kernel=6)["series"]
    dk = R.shift_table(st, wl.dms[:1])
    segs, idx, _ = R.all_segments(T, 1, windows, dk.max(axis=1))
    if len(segs):
        assert h.stage_times()["tree_tensor"] == 1
        assert_fit_match(st, vis, dk, segs, ser[0, 0][idx], R.fit_segments(st, vis, dk, segs))
    assert (ser == ser[:, :1]).all()
