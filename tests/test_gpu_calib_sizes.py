"""frbx_calibrate at the sizes where its kernels can go wrong: fewer APs than the 32 shares of the
sum, one more than a share, point counts that are no multiple of 32, the fewest and the most points
per channel, one channel, flagged points; and APs whose FP32 running sum overflows."""
import numpy as np
import pytest

from oracle import calib as K
from oracle import reference as R
import synth
from tests.test_gpu_calib import frbx  # noqa: F401
from tests.test_oracle_calib import _calibrator

pytestmark = pytest.mark.gpu


def _case(n_chan, n_point, l, seed):
    wl = synth.make_tiny(n_chan=n_chan, n_point=n_point, T=l + 3, n_bl=2, pulse=False, f_bw=16.0,
                         f0=800.0 + 16.0 * np.arange(n_chan))
    if n_point > 4:
        wl.flags = np.zeros(wl.C, np.uint8)
        wl.flags[[2, wl.C - 1]] = 1
    st = R.setup_from_workload(wl)
    rng = np.random.default_rng(seed)
    vis = np.stack([_calibrator(st, wl.T, 7.0 + b, rng.uniform(-3, 3, st.N), rng.uniform(-3, 3, st.N), noise=0.1, seed=b)
                    for b in range(2)])
    return wl, st, vis


@pytest.mark.parametrize("n_chan,n_point,l", [(3, 8, 1), (3, 8, 33), (5, 4, 31), (1, 256, 70), (7, 32, 64), (64, 16, 5)])
def test_sizes_match_the_oracle(frbx, n_chan, n_point, l):  # noqa: F811
    import torch
    wl, st, vis = _case(n_chan, n_point, l, 3)
    h = frbx.Handle.from_workload(wl)
    sbd, mbd, dl, ph = h.calibrate(torch.from_numpy(vis).cuda(), 2, l)
    for b in range(2):
        osbd, ombd, odl, oph = K.calibrate(st, vis[b], 2, l)
        assert (sbd[b], mbd[b]) == (osbd, ombd)
        # FP64 throughout: rounding (1e-15 of a grid step of 1000 / (8 f_bw) ns, a sum of 256 terms) far below
        np.testing.assert_allclose(dl[b], odl, atol=1e-9)
        np.testing.assert_allclose(np.angle(np.exp(1j * (ph[b] - oph))), 0.0, atol=1e-9)


def test_overflowing_shares_are_summed_in_fp64(frbx):  # noqa: F811
    """Two APs of one share near the largest float: their FP32 sum overflows, their FP64 sum does
    not, and a third AP of the opposite sign brings the total back into range."""
    import torch
    wl, st, vis = _case(3, 8, 80, 5)
    big = vis.copy()
    for k, v in ((2, 3e38), (34, 3e38), (66, -3e38)):  # APs 0, 32 and 64 of the segment
        big[:, k, 5] = v
    big[:, 3, 5] = -3e38
    h = frbx.Handle.from_workload(wl)
    got = h.calibrate(torch.from_numpy(big).cuda(), 2, 80)
    for b in range(2):
        want = K.calibrate(st, big[b], 2, 80)
        assert (got[0][b], got[1][b]) == tuple(want[:2])
        assert np.isfinite(got[2][b]).all()
        ok = np.arange(st.N) != 0  # channel 0's sum keeps rounding of 3e38
        np.testing.assert_allclose(got[2][b][ok], want[2][ok], atol=1e-9)
