"""What a batch object keeps between calls and reports: the captured graph when the DM trials that leave an AP change,
the time tile of setups fitted by the one-kernel window tree, and calls, of a batch or of one setup, that fail
while work is queued."""
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


def test_time_tile_of_the_one_kernel_tree(frbx):  # noqa: F811
    """Few series of a scan: k_tree16 takes its smallest tile, 128 APs, and that is what is reported."""
    wl = synth.make_small(T=1500, n_bl=2, dms=[0.0, 10.0])
    wl.pulses = []
    h = frbx.Handle.from_workload(wl)
    v = to_dev(synth.generate(wl))
    with frbx.Batch() as b:
        for _ in range(2):
            b.search([(h, v)], wl.dms, [2, 4])
            assert b.info()["time_tile"] == [128]
        assert b.info()["graph_captures"] == 1 and b.info()["graph_replays"] == 1


def test_failed_call_returns_after_its_work(frbx):  # noqa: F811
    """The second setup has no grid cell in the delay window, so the call fails after it queued the first one's shift
    table on a busy stream: it may return only when that stream is done."""
    import torch
    a, c = synth.make_small(T=300, n_bl=1, dms=[0.0]), synth.make_tiny(T=60, pulse=False)
    ha, hc = frbx.Handle.from_workload(a), frbx.Handle.from_workload(c)
    va, vc = to_dev(synth.generate(a)), to_dev(synth.generate(c))
    win = (15.0, 16.0)  # 15.6 ns is a cell of the first grid; the second one's cells are 31.25 ns apart
    st = torch.cuda.Stream()
    with frbx.Batch() as b:
        b.search([(ha, va)], [0.0], [2], sbd_win_ns=win)
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            torch.cuda._sleep(200_000_000)  # about 0.1 s
            with pytest.raises(frbx.FrbxError) as e:
                b.search([(ha, va), (hc, vc)], [0.0], [2], sbd_win_ns=win, stream=st)
            assert e.value.code == frbx.FRBX_EINVAL
            assert st.query()


def test_failed_calibration_returns_after_its_copy(frbx):  # noqa: F811
    """The scratch cap holds the cube but not the sums: the call fails with the cube's copy queued."""
    import torch
    wl = synth.make_small(T=300, n_bl=2, dms=[0.0])
    h = frbx.Handle.from_workload(wl)
    vis = torch.from_numpy(synth.generate(wl)).pin_memory()
    h.set_limits(scratch_cap_bytes=vis.numel() * 8 + 1024)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        torch.cuda._sleep(200_000_000)
        with pytest.raises(frbx.FrbxError) as e:
            h.calibrate(vis, 0, 200, stream=st)
        assert e.value.code == frbx.FRBX_ENOMEM
        assert st.query()
