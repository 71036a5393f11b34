"""Column blocks of the tensor-core window tree: 48 MBD columns per CTA (three epilogue warpgroups) or
32 (two), by the grid.  Grids whose columns are no multiple of 48 (the last block partly empty), the
smallest grids (32-column blocks), window sets with no anchor, with all anchors in tensor memory and
with two levels in shared memory, and MBD windows that touch one column of a block, cross a block's
edge or lie in the last, partly empty one.  Every segment against the FP64 oracle."""
import numpy as np
import pytest

import synth
from oracle import reference as R
from tests.gpu_helpers import assert_fit_match
from tests.test_gpu_tree import frbx, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu

# channel offsets (in units of the 16 MHz spacing) of grids with Lm 32, 64, 128, 256 and 512
GRIDS = {32: [0, 1, 9, 15], 64: [0, 7, 20, 31], 128: [0, 3, 33, 50, 63], 256: [0, 5, 64, 127], 512: [0, 11, 130, 255]}


def _wl(lm, T, windows):
    wl = synth.make_tiny(n_chan=len(GRIDS[lm]), n_point=64, T=T, n_bl=1, dms=(0.0, 30.0), windows=windows,
                         f0=3000.0 + 16.0 * np.array(GRIDS[lm], float))
    wl.pulses[0].width = 3
    return wl


def _check(frbx, wl, mbd=None):  # noqa: F811
    st = R.setup_from_workload(wl)
    vis = synth.generate(wl)
    h = frbx.Handle.from_workload(wl)
    out = h.search(to_dev(vis), wl.dms, wl.windows, want_series=True, kernel=6, mbd_win_ns=mbd)
    assert h.stage_times()["tree_tensor"] == 1
    dk = R.shift_table(st, wl.dms)
    segs, idx, _ = R.all_segments(wl.T, wl.n_bl, wl.windows, dk.max(axis=1))
    am, aq = R.window_masks(st, None, mbd)
    ref = R.fit_segments(st, vis, dk, segs, am, aq)
    flat = out["series"].reshape(-1)[idx]
    assert_fit_match(st, vis, dk, segs, flat, ref, (am, aq))
    assert aq[flat["mbd_idx"].astype(int)].all()
    return st


@pytest.mark.parametrize("lm", sorted(GRIDS))
def test_grids(frbx, lm):  # noqa: F811
    st = _check(frbx, _wl(lm, 150, [1, 2, 4, 8]))
    assert (st.Ls, st.Lm) == (128, lm)


@pytest.mark.parametrize("windows", [[1], [2], [1, 2, 4], [32, 1], [64, 2, 16]])
def test_anchor_levels(frbx, windows):  # noqa: F811
    _check(frbx, _wl(128, 190, windows))


@pytest.mark.parametrize("lo,hi", [(47, 47), (47, 48), (95, 96), (120, 127), (0, 0), (-3, 2)])
def test_mbd_windows(frbx, lo, hi):  # noqa: F811
    """Windows by MBD cell of the 256-column grid (cells of the second half are negative delays)."""
    wl = _wl(256, 100, [1, 2, 4])
    cell = 1000.0 / (256 * 16.0)
    for a, b in ((lo, hi), (-128 + lo, -128 + hi)) if lo >= 0 else ((lo, hi),):
        _check(frbx, wl, ((a - 0.25) * cell, (b + 0.25) * cell))
