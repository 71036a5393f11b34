"""The one-kernel window tree of 16-column MBD grids at the sizes where it can go wrong: 32, 64 and 128 SBD
rows (four, two and one time tile per CTA), fewer channels than slots, points that do not fill the
threads, scans shorter than a step, than a tile and just past one, DM trials that leave no or few APs, every
window level, and delay windows.  Every slot against the FP64 oracle."""
import numpy as np
import pytest

import synth
from oracle import reference as R
from tests.gpu_helpers import assert_fit_match
from tests.test_gpu_tree import frbx, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(frbx, n_chan, n_point, T, windows, dms=(0.0, 25.0), sbd=None, mbd=None, n_bl=2):  # noqa: F811
    wl = synth.make_tiny(n_chan=n_chan, n_point=n_point, T=T, n_bl=n_bl, dms=dms, windows=windows, f_bw=32.0, pulse=False,
                         f0=1400.0 + 32.0 * np.r_[0:n_chan - 1, 7])
    st = R.setup_from_workload(wl)
    assert (st.Ls, st.Lm) == (2 * n_point, 16)
    vis = synth.generate(wl)
    h = frbx.Handle.from_workload(wl)
    out = h.search(to_dev(vis), wl.dms, wl.windows, want_series=True, sbd_win_ns=sbd, mbd_win_ns=mbd)
    assert h.stage_times()["tree_tensor"] == 0
    dk = R.shift_table(st, wl.dms)
    segs, idx, _ = R.all_segments(wl.T, wl.n_bl, wl.windows, dk.max(axis=1))
    empty = np.ones(out["series"].size, bool)
    empty[idx] = False
    assert (out["series"].reshape(-1)["amp"][empty] == -1.0).all()
    if len(segs) == 0:
        return
    assert h.stage_times()["tree_chunks"] == 1
    am, aq = R.window_masks(st, sbd, mbd)
    ref = R.fit_segments(st, vis, dk, segs, am, aq)
    flat = out["series"].reshape(-1)[idx]
    assert_fit_match(st, vis, dk, segs, flat, ref, (am, aq))


@pytest.mark.parametrize("n_chan,n_point", [(8, 16), (8, 32), (8, 64), (3, 32), (5, 16), (3, 64)])
def test_shapes(frbx, n_chan, n_point):  # noqa: F811
    _check(frbx, n_chan, n_point, 261, [1, 2, 4, 8, 16])


@pytest.mark.parametrize("T", [1, 2, 3, 4, 63, 127, 128, 129, 257, 1153])
def test_scan_lengths(frbx, T):  # noqa: F811
    _check(frbx, 8, 32, T, [1, 2, 8] if T < 200 else [2, 16], dms=(0.0, 25.0, 2000.0), n_bl=1)


@pytest.mark.parametrize("windows", [[1], [2], [4], [8, 1], [32, 64], [64, 16, 2]])
def test_levels(frbx, windows):  # noqa: F811
    _check(frbx, 8, 32, 300, windows, n_bl=1)


@pytest.mark.parametrize("n_point", [16, 32, 64])
@pytest.mark.parametrize("sbd,mbd", [((-70.0, 90.0), None), (None, (-6.0, 4.5)), ((100.0, 240.0), (1.9, 2.0))])
def test_delay_windows(frbx, n_point, sbd, mbd):  # noqa: F811
    _check(frbx, 8, n_point, 150, [1, 2, 4, 8], sbd=sbd, mbd=mbd, n_bl=1)
