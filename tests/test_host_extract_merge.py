"""The DM merge of many pulses, which is split over threads by series: one window is enough for a pulse, so thousands of
them, spread over series, all in one series, or in one of several.  Against the oracle's single pass (no GPU)."""
import numpy as np
import pytest

from tests.test_host_extract import compare, frbx, random_events, to_events  # noqa: F401


@pytest.mark.parametrize("n_series,n_dm,heavy", [(6, 30, None), (1, 60, None), (5, 60, 2), (3, 60, 0)])
def test_many_pulses(frbx, n_series, n_dm, heavy):  # noqa: F811
    rng = np.random.default_rng(n_series)
    windows, T, Lm = [1], 300, 16
    cands = random_events(rng, n_series, n_dm, windows, T, Lm, 0.4)
    if heavy is not None:  # the other series nearly empty
        cands = [c for c in cands if c["series"] == heavy or rng.random() < 0.01]
    assert len(cands) > 6000  # one-AP windows: every event is a pulse, in groups of its own per DM trial
    assert compare(frbx, to_events(cands, frbx), n_series, T, n_dm, windows, Lm, 1, use_mbd=False, cross=True) > 0
