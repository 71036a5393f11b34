"""The choice of column blocks of the tensor-core window tree: 32 MBD columns per CTA where the launch is small, 48
where it takes rounds of CTAs fewer.  The same DM trial a few times and many times over, so that one search of each
pair takes either form: every series has to be the same bits, and the first one is checked against the FP64 oracle."""
import numpy as np
import pytest

import synth
from oracle import reference as R
from tests.gpu_helpers import assert_fit_match
from tests.test_gpu_tree import frbx, to_dev  # noqa: F401
from tests.test_gpu_tree_cols import GRIDS

pytestmark = pytest.mark.gpu


def _check(frbx, lm, T, windows, sbd=None, mbd=None, kernel=6, oracle=True):  # noqa: F811
    wl = synth.make_tiny(n_chan=len(GRIDS[lm]), n_point=64, T=T, n_bl=1, dms=(0.0,), windows=windows,
                         f0=3000.0 + 16.0 * np.array(GRIDS[lm], float))
    vis = synth.generate(wl)
    vd = to_dev(vis)
    h = frbx.Handle.from_workload(wl)
    kw = dict(want_series=True, kernel=kernel, sbd_win_ns=sbd, mbd_win_ns=mbd)
    few = h.search(vd, np.zeros(2), windows, **kw)["series"]
    many = h.search(vd, np.zeros(500), windows, **kw)["series"]
    assert h.stage_times()["tree_tensor"] == 1
    assert (few == few[:, :1]).all() and (many == few[:, :1]).all()
    if oracle:
        st = R.setup_from_workload(wl)
        dk = R.shift_table(st, wl.dms)
        segs, idx, _ = R.all_segments(T, 1, windows, dk.max(axis=1))
        am, aq = R.window_masks(st, sbd, mbd)
        assert_fit_match(st, vis, dk, segs, few[0, 0][idx], R.fit_segments(st, vis, dk, segs, am, aq), (am, aq))


@pytest.mark.parametrize("lm", [128, 256, 512])
@pytest.mark.parametrize("windows", [[1, 2, 4, 8], [2, 16], [1], [64, 4]])
def test_whole_grid(frbx, lm, windows):  # noqa: F811
    _check(frbx, lm, 90, windows)


@pytest.mark.parametrize("kernel", [7, 8])
def test_one_product_forms(frbx, kernel):  # noqa: F811
    _check(frbx, 256, 90, [1, 2, 4, 8], kernel=kernel, oracle=False)


@pytest.mark.parametrize("sbd", [100.0, 400.0, 800.0, 1500.0])
def test_delay_windows(frbx, sbd):  # noqa: F811
    """SBD cells of 31.25 ns: 16, 32 and 64 rows, and more than half of the 128."""
    _check(frbx, 256, 300, [1, 2, 4, 8], sbd=(-sbd, sbd))


def test_mbd_window_across_an_edge(frbx):  # noqa: F811
    cell = 1000.0 / (256 * 16.0)
    _check(frbx, 256, 90, [1, 2, 4], mbd=(46.75 * cell, 48.25 * cell))
