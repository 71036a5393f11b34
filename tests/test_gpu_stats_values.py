"""Normalised power and crossings where the float-pair arithmetic of the normalisation is at its limits: series
whose amplitudes differ by so little that FP32 squares of the differences vanish, or by little more than a float
resolves, the rounding of P, and amplitudes that are not finite.  P is recomputed in FP64 from the amplitudes the search returns."""
import numpy as np
import pytest

import synth
from tests.test_gpu_stats import _check, _run
from tests.test_gpu_tree import frbx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-21, 1e-20, 1e-19])
def test_differences_whose_squares_underflow(frbx, scale):  # noqa: F811
    """Amplitudes near 50 x scale that vary by 1e-4 of themselves."""
    def edit(vis):
        rng = np.random.default_rng(3)
        vis[:] = vis[:, :1] * (scale * (1.0 + 1e-4 * rng.standard_normal((vis.shape[0], vis.shape[1], 1)))).astype(np.float32)
    out, combos, off = _run(frbx, 200, edit)
    _check(out, combos, off)
    assert out["counts"]["events"] > 0


def test_differences_that_cancel(frbx):  # noqa: F811
    """Two slots each: where their middle is a float, the differences from it add up to zero, and their squares
    vanish in FP32."""
    def edit(vis):
        vis[:, 0] *= np.float32(1e-21)
        rng = np.random.default_rng(4)
        vis[:, 1] = vis[:, 0] * (1.0 + 1e-4 * rng.uniform(0.5, 2.0, (vis.shape[0], 1))).astype(np.float32)
    out, combos, off = _run(frbx, 2, edit, n_bl=32, windows=(1,))
    amp = out["series"]["amp"][:, 0]
    assert ((amp[:, 1] - amp[:, 0]) ** 2 == 0).all() and (amp[:, 0] != amp[:, 1]).sum() > 16
    _check(out, combos, off)
    assert (np.abs(out["pnorm"][:, 0]) == (amp[:, :1] != amp[:, 1:])).all()


def test_p_is_the_fp64_expression_rounded(frbx):  # noqa: F811
    """Every slot made a crossing: the events hold (A - mean) / std in FP64, rounded, and so does P.  The first slots
    lie several std above the mean."""
    import torch
    n_bl, T = 48, 8192
    wl = synth.make_small(T=T, n_bl=n_bl, dms=np.arange(10.0))
    gen = torch.Generator("cuda").manual_seed(5)
    vis = torch.view_as_complex(torch.randn((n_bl, T, wl.C, 2), device="cuda", generator=gen))
    vis[:, :60] *= 1.3
    out = frbx.Handle.from_workload(wl).search(vis, wl.dms, [1], threshold=-100.0, nwin_min=2, want_series=True,
                                               want_events=True)
    ev = out["events"]
    assert len(ev) == (out["series"]["amp"] >= 0).sum() > 3_900_000
    assert np.array_equal(ev["pnorm"], out["pnorm"][ev["series"], ev["dm_idx"], ev["k0"]])


@pytest.mark.parametrize("part", [1e-4, 1e-6, 2e-7])
def test_nearly_constant_series(frbx, part):  # noqa: F811
    """Amplitudes that vary by little more than a float resolves, alone and in combinations."""
    def edit(vis):
        rng = np.random.default_rng(6)
        vis[:] = vis[:, :1] * (1.0 + part * rng.standard_normal((vis.shape[0], vis.shape[1], 1))).astype(np.float32)
    out, combos, off = _run(frbx, 300, edit)
    _check(out, combos, off)
    assert out["counts"]["events"] > 0


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_not_finite_amplitudes(frbx, value):  # noqa: F811
    """The FP64 expression of a series with such an amplitude has a mean and std that are not finite, and
    std > 0 decides: P and the crossings are those of the expression, also of combinations that hold it."""
    def edit(vis):
        vis[1, 50, 7] = value
    out, combos, off = _run(frbx, 100, edit)
    ref, _, _ = _run(frbx, 100)
    amp = out["series"]["amp"].astype(np.float64)
    n_base = out["counts"]["events_baseline"]
    base, comb = out["events"][:n_base], out["events"][n_base:]
    touched = 0
    for d in range(2):
        for w in range(3):
            a = amp[1, d, off[w]:off[w + 1]]
            a = a[~(a < 0)]
            with np.errstate(invalid="ignore"):
                mean = a.mean()
                sd = np.sqrt(((a - mean) ** 2).mean())
                p = (a - mean) / sd if sd > 0 else np.zeros_like(a)
            if np.isfinite(a).all():
                continue
            touched += 1
            np.testing.assert_array_equal(out["pnorm"][1, d, off[w]:off[w] + a.size], p.astype(np.float32))
            assert not ((base["series"] == 1) & (base["dm_idx"] == d) & (base["win_idx"] == w)).any()
            # both combinations hold baseline 1 or not: 0b111 does, 0b101 does not
            assert not ((comb["series"] == 0) & (comb["dm_idx"] == d) & (comb["win_idx"] == w)).any()
    assert touched > 0
    for s in (0, 2):
        assert np.array_equal(out["pnorm"][s], ref["pnorm"][s])
    rb = ref["events"][:ref["counts"]["events_baseline"]]
    rc = ref["events"][ref["counts"]["events_baseline"]:]
    assert np.array_equal(base[base["series"] != 1], rb[rb["series"] != 1])
    assert np.array_equal(comb[comb["series"] == 1], rc[rc["series"] == 1])
