"""What a call may need: a setup whose tables fill the shared memory of the per-segment FFT fit, and a scratch cap
that holds a search's series, tables and events and nothing more."""
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


@pytest.mark.parametrize("n_dm,windows,combos,thr", [(7, [3, 5, 9], [], 2.5), (3000, [2], [], 2.5), (50, [1, 3], [3], 2.5),
                                                     (50, [1, 3], [3, 2], -0.5)])
def test_scratch_cap_of_series_tables_and_events(frbx, n_dm, windows, combos, thr):  # noqa: F811
    wl = synth.make_small(T=300, n_bl=2, dms=np.linspace(0.0, 50.0, n_dm))
    wl.pulses = []
    vis = synth.generate(wl)
    vis[0, 200:] = 0  # equal amplitudes in part of a series
    vd = to_dev(vis)
    kw = dict(threshold=thr, want_events=True, kernel=1, combos=combos)
    ref = frbx.Handle.from_workload(wl).search(vd, wl.dms, windows, **kw)
    n_base, n_ev = ref["counts"]["events_baseline"], ref["counts"]["events"]
    assert n_base > 0
    ns = max(wl.n_bl, len(combos)) * n_dm * len(windows)
    # shift table, series, mean and std, counts, offsets, events, DM list / window tables, largest shifts, combinations
    need = [4 * n_dm * wl.C, 8 * wl.n_bl * n_dm * ref["S_tot"], 16 * ns, 4 * (ns + 1), 8 * (ns + 1),
            32 * max(n_base, n_ev - n_base), max(8 * n_dm, 4 * (48 + n_dm * len(windows))) + 4096, 4 * n_dm]
    need += [8 * len(combos)] * bool(combos)
    h = frbx.Handle.from_workload(wl)
    h.set_limits(scratch_cap_bytes=sum(max(256, b) for b in need))
    for _ in range(2):
        out = h.search(vd, wl.dms, windows, **kw)
        assert np.array_equal(out["events"], ref["events"]) and np.array_equal(out["pulses"], ref["pulses"])
    # less than the series alone is refused
    h2 = frbx.Handle.from_workload(wl)
    h2.set_limits(scratch_cap_bytes=7 * wl.n_bl * n_dm * ref["S_tot"])
    with pytest.raises(frbx.FrbxError) as e:
        h2.search(vd, wl.dms, windows, **kw)
    assert e.value.code == frbx.FRBX_ENOMEM
