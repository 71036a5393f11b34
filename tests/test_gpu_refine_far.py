"""Refinement windows that start far before the cube, where a sample's phase factor f0 t_ap (u + i) is the small
difference of large terms, and positions that no integer holds."""
import numpy as np
import pytest

import synth
from tests.test_gpu_refine import frbx  # noqa: F401

pytestmark = pytest.mark.gpu


def test_rate_gradient_of_windows_that_start_before_the_cube(frbx):  # noqa: F811
    """Two channels with one used point each, a cube that is 1 (i) at AP 1 of the first (second) and zero
    elsewhere, windows that reach it from up to a million APs before: the one sample with a value has u + i = 1, so
    the rate's gradient is 2 2 pi 1e-6 (f0_1 - f0_0) of the FP32-rounded f0 t_ap, whatever the start.  f0 lies
    2^-38 of itself above the middle of two floats; the SBD delay turns the used points by a quarter (a phase of zero
    would be evaluated in FP64 as it is)."""
    import torch
    f0 = 1400.0 + 2.0 ** -14 + 1400.0 * 2.0 ** -38
    wl = synth.make_tiny(n_chan=2, n_point=2, T=8, n_bl=1, dms=(0.0,), f0=[f0, f0 + 32.0], f_bw=32.0, pulse=False)
    h = frbx.Handle.from_workload(wl)
    vis = np.zeros((1, 8, 4), np.complex64)
    vis[0, 1, 1], vis[0, 1, 3] = 1.0, 1.0j
    rng = np.random.default_rng(0)
    start = np.r_[rng.integers(-5, 5, 16), -rng.integers(10, 1000, 240), -rng.integers(10 ** 4, 10 ** 6, 1792)]
    start = np.minimum(start, 1)
    th = np.zeros((start.size, 5))
    th[:, 1], th[:, 2] = start, 15.625
    width = (4 - start).astype(np.int32)
    vd, pt, wt = torch.from_numpy(vis).cuda(), torch.from_numpy(th).cuda(), torch.from_numpy(width).cuda()
    power, g, status = frbx.refine_power(h, vd, pt, wt)
    dpar = frbx.refine_adjoint(h, vd, pt, wt, g, torch.ones(start.size, device="cuda")).cpu().numpy()
    assert (power.cpu().numpy() == 2.0).all()
    f = np.float32
    fx = np.array([f0, f0 + 32.0]).astype(f)
    want = f(f(f(2.0) * f(6.283185307179586)) * f(1e-6)) * f(fx[1] - fx[0])
    assert np.array_equal(dpar[:, 4].astype(f), np.full(start.size, want, f))


def test_positions_that_no_integer_holds(frbx):  # noqa: F811
    import torch
    wl = synth.make_small(T=400, n_bl=2, dms=[300.0])
    h = frbx.Handle.from_workload(wl)
    t0 = [np.nan, np.inf, -np.inf, 1e300, -1e300, 2.0 ** 30, -2.0 ** 30, 2.0 ** 30 - 0.5, -2.0 ** 30 + 0.5, 2147483646.5,
          2147483647.0, 2147483647.9999998, 2147483648.0, -2147483648.0, -2147483649.5, 4294967297.0, -4294967295.0]
    th = np.zeros((len(t0) + 2, 8))
    th[:len(t0), 1] = t0
    th[len(t0):, 0] = [np.nan, np.inf]
    th[len(t0):, 1] = 50.0
    width = np.full(len(th), 8, np.int32)
    vd, pt, wt = torch.from_numpy(synth.generate(wl)).cuda(), torch.from_numpy(th).cuda(), torch.from_numpy(width).cuda()
    power, g, status = frbx.refine_power(h, vd, pt, wt)
    dpar = frbx.refine_adjoint(h, vd, pt, wt, g, torch.ones(len(th), device="cuda")).cpu().numpy()
    assert (status.cpu().numpy() == 1).all() and (power.cpu().numpy() == 0).all()
    assert (dpar == 0).all()
