"""Refinement at the sizes where its kernels can go wrong: few and many candidates and baselines, windows
longer than the taps loaded ahead and of a single AP, candidates whose taps leave the
cube at either end, whole cycles of rate per AP, large delays, and parameters that are not finite.
Forward and adjoint against the FP64 oracle with the tolerances of test_gpu_refine."""
import numpy as np
import pytest

import synth
from oracle import reference as R
from oracle import refine as F
from tests.test_gpu_refine import _random_params, frbx  # noqa: F401

pytestmark = pytest.mark.gpu


def _case(n_bl, seed):
    wl = synth.make_small(T=400, n_bl=n_bl, dms=[300.0])
    wl.pulses = []
    wl.flags = np.zeros(wl.C, np.uint8)
    wl.flags[[3, 40, 255]] = 1
    return wl, R.setup_from_workload(wl), synth.generate(wl), np.random.default_rng(seed)


def _run(frbx, wl, vis, th, width):  # noqa: F811
    import torch
    h = frbx.Handle.from_workload(wl)
    vd, pt, wt = torch.from_numpy(vis).cuda(), torch.from_numpy(th).cuda(), torch.from_numpy(width).cuda()
    power, g, status = frbx.refine_power(h, vd, pt, wt)
    dpar = frbx.refine_adjoint(h, vd, pt, wt, g, torch.ones(len(th), device="cuda"))
    return power.cpu().numpy(), status.cpu().numpy(), dpar.cpu().numpy()


def _compare(st, vis, th, width, P, dpar):
    for i in range(len(th)):
        Po, Go = F.coherent_power(st, vis, th[i], int(width[i]))[:2]
        assert P[i] == pytest.approx(Po, rel=1e-4)
        Go = np.asarray(Go)
        for k0 in range(5):  # by parameter type: DM, t0, then tau_s, tau_m, rho of every baseline
            ks = [k0] if k0 < 2 else list(range(k0, len(Go), 3))
            np.testing.assert_allclose(dpar[i][ks], Go[ks], atol=2e-3 * np.abs(Go[ks]).max())


@pytest.mark.parametrize("n_bl,n_cand", [(1, 3), (3, 2), (5, 320), (4, 640)])
def test_counts(frbx, n_bl, n_cand):  # noqa: F811
    wl, st, vis, rng = _case(n_bl, n_cand)
    th = _random_params(rng, wl, n_cand)
    th[:, 0] *= 0.3
    th[:, 1] = rng.uniform(2.0, 150.0, n_cand)
    width = rng.choice([1, 2, 3, 8, 37], n_cand).astype(np.int32)
    P, status, dpar = _run(frbx, wl, vis, th, width)
    assert not status.any()
    pick = np.r_[0:min(3, n_cand), n_cand - 2:n_cand]
    _compare(st, vis, th[pick], width[pick], P[pick], dpar[pick])


def test_rates_and_delays_of_many_cycles(frbx):  # noqa: F811
    """rho of 1e3 to 3e3 is 1.4 to 5 cycles per AP, delays of 1e6 ns thousands of cycles: the phases are
    reduced before they are rounded, so the forward tolerance does not change.  The gradient of a rate
    and of t0 has terms of the rate itself, the tolerance by type holds for it too."""
    wl, st, vis, rng = _case(3, 9)
    th = _random_params(rng, wl, 4)
    th[:, 0] *= 0.2
    th[:, 1] = rng.uniform(20.0, 100.0, 4)
    th[:, 2::3] += 1e6
    th[:, 3::3] -= 1e6
    th[:, 4::3] = rng.uniform(1e3, 3e3, (4, 3)) * rng.choice([-1.0, 1.0], (4, 3))
    width = np.array([1, 4, 8, 16], np.int32)
    P, status, dpar = _run(frbx, wl, vis, th, width)
    _compare(st, vis, th, width, P, dpar)


def test_edges_and_values_that_are_not_finite(frbx):  # noqa: F811
    wl, st, vis, rng = _case(2, 11)
    th = _random_params(rng, wl, 9)
    th[:, 0] = 10.0
    th[:, 1] = [0.5, 1.0, 390.0, -50.0, 1e12, np.nan, np.inf, 100.0, 100.0]
    th[7, 2] = np.nan
    th[8, 7] = np.inf
    width = np.full(9, 8, np.int32)
    P, status, dpar = _run(frbx, wl, vis, th, width)
    assert status.tolist() == [1, 0, 1, 1, 1, 1, 1, 0, 0]
    _compare(st, vis, th[1:2], width[1:2], P[1:2], dpar[1:2])
    assert (P[3:7] == 0).all() and np.isnan(P[7]) and np.isnan(P[8])
