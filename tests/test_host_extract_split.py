"""The split of the host extraction over threads, which cuts event lists between (series, DM trial)s: lists
of a few thousand events whose cuts fall inside a series, runs of DM trials without events, one DM
trial that holds nearly all of them, and MBD cells whose angle from the mean is a quarter turn or near half
a turn.  Against the oracle's single pass (no GPU)."""
import numpy as np
import pytest

from tests.test_host_extract import compare, frbx, random_events, to_events  # noqa: F401


@pytest.mark.parametrize("n_series,n_dm,density,skew", [(1, 40, 0.2, 0), (2, 25, 0.25, 0), (3, 9, 0.3, 7), (1, 3, 0.6, 2)])
def test_cuts_inside_a_series(frbx, n_series, n_dm, density, skew):  # noqa: F811
    rng = np.random.default_rng(n_dm)
    windows, T, Lm = [2, 4, 8, 16], 260, 16
    cands = random_events(rng, n_series, n_dm, windows, T, Lm, density)
    if skew:  # DM trials 0 .. skew - 1 nearly empty
        cands = [c for c in cands if c["d"] >= skew or rng.random() < 0.02]
    cands = [c for c in cands if c["d"] % 5 != 3]
    ev = to_events(cands, frbx)
    n = compare(frbx, ev, n_series, T, n_dm, windows, Lm, 2, use_mbd=True, cross=True)
    n += compare(frbx, ev, n_series, T, n_dm, windows, Lm, 2, use_mbd=False, cross=False)
    assert n > 0


@pytest.mark.parametrize("cells", [(0, 4, 12), (0, 8), (15, 1, 7, 9), (8, 0, 0), (4, 4, 12, 12, 0)])
def test_angles_at_the_quarter_and_half_turn(frbx, cells):  # noqa: F811
    windows = [1, 2, 4, 8, 16]
    cands = [dict(series=0, d=0, w=i % 5, k0=16, amp=1.0, p=float(np.float32(4 + 0.25 * i)), m=0, q=q)
             for i, q in enumerate(cells)]
    compare(frbx, to_events(cands, frbx), 1, 64, 1, windows, 16, 1, use_mbd=True, cross=True)
