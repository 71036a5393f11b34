"""Packed delay windows of the tensor-core tree: searched SBD rows that fit 16, 32 or 64 tile rows, so that one
CTA walks eight, four or two time tiles (16 lanes, a row quarter or a pair of them each), on scans that
leave the last pieces short or empty and DM trials that end tiles early.  Every slot against the FP64
oracle; the one-product forms (kernels 7 and 8) against the same search in FP32 (kernel 4)."""
import numpy as np
import pytest

import synth
from oracle import reference as R
from tests.gpu_helpers import assert_fit_match
from tests.test_gpu_tree import frbx, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu

# SBD windows (ns) by the tile rows they take at 15.6 ns a cell, rotated to a multiple of 8
ROWS = {16: (-64.0, 64.0), 9: (0.0, 130.0), 32: (-200.0, 200.0), 64: (-450.0, 420.0)}


def _wl(T, dms=(0.0, 60.0, 900.0)):
    wl = synth.make_vgos(T=T, n_bl=1, n_dm=len(dms))
    wl.dms = np.array(dms)
    wl.pulses = []
    wl.windows = [1, 2, 4, 8, 16, 32]
    return wl


@pytest.mark.parametrize("rows", sorted(ROWS))
@pytest.mark.parametrize("T", [33, 128, 515, 1100])
def test_every_slot(frbx, rows, T):  # noqa: F811
    wl = _wl(T)
    st = R.setup_from_workload(wl)
    vis = synth.generate(wl)
    h = frbx.Handle.from_workload(wl)
    out = h.search(to_dev(vis), wl.dms, wl.windows, want_series=True, sbd_win_ns=ROWS[rows])
    assert h.stage_times()["tree_tensor"] == 1
    dk = R.shift_table(st, wl.dms)
    segs, idx, _ = R.all_segments(wl.T, 1, wl.windows, dk.max(axis=1))
    am, aq = R.window_masks(st, ROWS[rows], None)
    ref = R.fit_segments(st, vis, dk, segs, am, aq)
    flat = out["series"].reshape(-1)[idx]
    assert_fit_match(st, vis, dk, segs, flat, ref, (am, aq))
    empty = np.ones(out["series"].size, bool)
    empty[idx] = False
    assert (out["series"].reshape(-1)["amp"][empty] == -1.0).all()


@pytest.mark.parametrize("kernel,tol", [(7, 1e-2), (8, 1.2e-1)])
@pytest.mark.parametrize("rows", [16, 32])
def test_one_product_forms(frbx, kernel, tol, rows):  # noqa: F811
    """BF16 rounds each operand by 2^-9, E4M3 by 2^-4: the tolerances on |G| of the whole-tile forms."""
    wl = _wl(700)
    vd = to_dev(synth.generate(wl))
    h = frbx.Handle.from_workload(wl)
    a = h.search(vd, wl.dms, wl.windows, want_series=True, sbd_win_ns=ROWS[rows], kernel=kernel)["series"]["amp"]
    b = h.search(vd, wl.dms, wl.windows, want_series=True, sbd_win_ns=ROWS[rows], kernel=4)["series"]["amp"]
    ok = b >= 0
    assert np.array_equal(ok, a >= 0)
    assert (np.abs(a - b)[ok] <= tol * b[ok]).all()
