"""Normalisation and threshold (Eq. 6) at the sizes and values where the kernels can go wrong: slot counts
around the 32 of a hit word and the 256 of a CTA, series whose first amplitude lies far from the mean,
constant series, amplitudes whose squares FP32 cannot hold, values that are not finite, and baseline
combinations.  P and the crossings are recomputed in FP64 from the amplitudes the search returns."""
import numpy as np
import pytest

import synth
from tests.test_gpu_tree import frbx  # noqa: F401

pytestmark = pytest.mark.gpu

THR = 2.5


def _run(frbx, T, edit=None, n_bl=3, windows=(1, 2, 4)):  # noqa: F811
    import torch
    wl = synth.make_small(T=T, n_bl=n_bl, dms=np.array([0.0, 30.0]))
    wl.pulses = []
    vis = synth.generate(wl)
    if edit is not None:
        edit(vis)
    h = frbx.Handle.from_workload(wl)
    combos = [0b111, 0b101]
    out = h.search(torch.from_numpy(vis).cuda(), wl.dms, list(windows), threshold=THR, combos=combos, want_series=True,
                   want_events=True)
    off, _ = frbx.frbx_series_layout(T, np.array(windows, np.int32))
    return out, combos, list(off) + [out["S_tot"]]


def _check(out, combos, off):
    """P of every valid slot to FP32 rounding of the FP64 value (the sums' error is 1e-13 of it), and the
    crossings wherever P is not within 1e-8 of the threshold."""
    amp = out["series"]["amp"].astype(np.float64)
    n_bl, n_dm, _ = amp.shape
    groups = [(b, 1 << b) for b in range(n_bl)] + [(n_bl + i, m) for i, m in enumerate(combos)]
    ev = out["events"]
    n_base = out["counts"]["events_baseline"]
    got = {}
    for i, e in enumerate(ev):
        s = int(e["series"]) + (n_bl if i >= n_base else 0)
        got.setdefault((s, int(e["dm_idx"]), int(e["win_idx"])), []).append(e)
    order = [(s, d, w) for s, _ in groups for d in range(n_dm) for w in range(len(off) - 1)]
    assert [k for k in order if k in got] == list(got)  # events in order
    for s, mask in groups:
        for d in range(n_dm):
            for w in range(len(off) - 1):
                a = sum(amp[b, d, off[w]:off[w + 1]] for b in range(n_bl) if mask >> b & 1)
                valid = amp[0, d, off[w]:off[w + 1]] >= 0
                a = a[valid]
                sd = a.std() if a.size else 0.0
                p = (a - a.mean()) / sd if sd > 0 else np.zeros_like(a)
                if s < n_bl:
                    np.testing.assert_allclose(out["pnorm"][s, d, off[w]:off[w + 1]][valid], p, rtol=2.0 ** -23, atol=1e-12)
                k = got.get((s, d, w), [])
                step = max(1, (1, 2, 4, 8)[w] // 2)
                hit = {int(e["k0"]) // step: e for e in k}
                sure = np.abs(p - THR) > 1e-8
                assert all((i in hit) == (p[i] > THR) for i in np.flatnonzero(sure))
                for i, e in hit.items():
                    assert e["amp"] == np.float32(a[i]) and abs(e["pnorm"] - p[i]) <= 2.0 ** -23 * abs(p[i])


@pytest.mark.parametrize("T", [6, 31, 32, 33, 65, 257, 1030])
def test_slot_counts(frbx, T):  # noqa: F811
    _check(*_run(frbx, T))


@pytest.mark.parametrize("scale", [1e-14, 1e-6, 1e9, 1e14])
def test_scales(frbx, scale):  # noqa: F811
    def edit(vis):
        vis *= np.float32(scale)
    _check(*_run(frbx, 200, edit))


def test_first_slots_far_from_the_mean(frbx):  # noqa: F811
    def edit(vis):
        vis[:, :1] *= 1e5
    _check(*_run(frbx, 400, edit))


def test_constant_and_empty_series(frbx):  # noqa: F811
    def edit(vis):
        vis[0] = vis[0, :1]  # the same spectrum at every AP
        vis[1] = 0
    out, combos, off = _run(frbx, 100, edit)
    assert (out["pnorm"][0, 0] == 0).all() and (out["pnorm"][1] == 0).all()
    assert not any(e["series"] == 0 and e["dm_idx"] == 0 for e in out["events"][:out["counts"]["events_baseline"]])


def test_values_that_are_not_finite(frbx):  # noqa: F811
    def edit(vis):
        vis[1, 50, 7] = np.inf
    out, combos, off = _run(frbx, 100, edit)
    ok = out["events"][:out["counts"]["events_baseline"]]
    assert (out["pnorm"][1] == 0).all() or np.isfinite(out["pnorm"][1]).all()
    assert not (ok["series"] == 1).any() or np.isfinite(ok["pnorm"]).all()
    ref, _, _ = _run(frbx, 100)
    for s in (0, 2):
        assert np.array_equal(out["pnorm"][s], ref["pnorm"][s])
