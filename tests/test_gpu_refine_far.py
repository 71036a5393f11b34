"""Refinement at positions that no integer holds."""
import numpy as np
import pytest

import synth
from tests.test_gpu_refine import frbx  # noqa: F401

pytestmark = pytest.mark.gpu


def test_positions_that_no_integer_holds(frbx):  # noqa: F811
    import torch
    wl = synth.make_small(T=400, n_bl=2, dms=[300.0])
    h = frbx.Handle.from_workload(wl)
    t0 = [np.nan, np.inf, -np.inf, 1e300, -1e300, 2.0 ** 30, -2.0 ** 30, 2.0 ** 30 - 0.5, -2.0 ** 30 + 0.5, 2147483646.5, 2147483647.0, 2147483647.9999998, 2147483648.0, -2147483648.0,
          -2147483649.5, 4294967297.0, -4294967295.0]
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
