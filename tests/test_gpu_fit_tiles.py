"""Segment lists and per-segment searches of sizes that take other tiles: one 512-thread CTA per
segment (lists up to two segments per SM), one 128-thread CTA per segment, several segments per
CTA with a ragged last one, and short time tiles of a small search.  A segment's result does not
depend on the list it is in, and sampled rows match the FP64 oracle."""
import numpy as np
import pytest

import synth
from oracle import reference as R
from tests.gpu_helpers import assert_fit_match

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def frbx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_02391_gb300 import _build
    _build.build()
    from paper_1801_02391_gb300 import frbx as f
    f.load()
    return f


@pytest.mark.parametrize("setup", ["vgos", "small", "c1024"])
def test_lists_of_every_tile(frbx, setup):
    import torch
    if setup == "vgos":
        wl = synth.make_vgos(T=120, n_bl=2, n_dm=3)
        wl.dms = np.array([0.0, 20.0, 60.0])
    elif setup == "small":
        wl = synth.make_small(T=160, n_bl=2, dms=np.array([0.0, 20.0, 60.0]))
    else:
        wl = synth._batch_setup("c1024", 43, 120, 2, [0.0, 20.0, 60.0])
    wl.pulses = []
    st = R.setup_from_workload(wl)
    vis = synth.generate(wl)
    vd = torch.from_numpy(vis).cuda()
    dk = R.shift_table(st, wl.dms)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(4)
    n = 2 * 8 * 4 * sms + 5  # two segments per CTA, the last one alone
    rows = np.zeros((n, 4), np.int32)
    rows[:, 0] = rng.integers(0, 2, n)
    rows[:, 1] = rng.integers(0, 3, n)
    rows[:, 2] = rng.choice([1, 2, 3, 7, 16], n)
    rows[:, 3] = rng.integers(0, wl.T - dk.max(axis=1)[rows[:, 1]] - rows[:, 2] + 1)
    h = frbx.Handle.from_workload(wl)
    whole = h.fit_segments(vd, wl.dms, rows)
    for m in (1, 2 * sms, 2 * sms + 1, 8 * 4 * sms + 1):
        assert np.array_equal(h.fit_segments(vd, wl.dms, rows[:m]), whole[:m])
    pick = np.concatenate([np.arange(12), np.arange(n - 12, n)])
    ref = R.fit_segments(st, vis, dk, rows[pick])
    assert_fit_match(st, vis, dk, rows[pick], whole[pick], ref)


def test_search_of_short_time_tiles(frbx):
    """Windows that are no powers of two on one baseline: the time tile shrinks to fill the GPU,
    and every slot equals the same segment fitted from a list."""
    import torch
    wl = synth.make_vgos(T=203, n_bl=1, n_dm=2)
    wl.dms = np.array([0.0, 40.0])
    wl.pulses = []
    st = R.setup_from_workload(wl)
    vis = synth.generate(wl)
    vd = torch.from_numpy(vis).cuda()
    windows = [3, 6, 10]
    h = frbx.Handle.from_workload(wl)
    out = h.search(vd, wl.dms, windows, want_series=True)
    segs, idx, _ = R.all_segments(wl.T, 1, windows, R.shift_table(st, wl.dms).max(axis=1))
    assert np.array_equal(out["series"].reshape(-1)[idx], h.fit_segments(vd, wl.dms, np.asarray(segs, np.int32)))
