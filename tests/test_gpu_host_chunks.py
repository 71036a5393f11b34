"""Chunks of a search of host input: several baselines each where one would leave the GPU idle, one each where it fills
the GPU, and the same results as from device memory."""
import numpy as np
import pytest

import synth
from tests.test_gpu_tree import frbx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bl,n_dm,T,most", [(15, 2, 300, 4), (8, 2, 600, 4), (3, 1, 40, 1), (2, 16, 1100, 2)])
def test_host_input_chunks(frbx, n_bl, n_dm, T, most):  # noqa: F811
    """Chunks that fill the GPU: several baselines with few DM trials, one baseline with many."""
    import torch
    wl = synth.make_vgos(T=T, n_bl=n_bl, n_dm=n_dm)
    wl.dms = np.linspace(0.0, 20.0, n_dm)
    wl.pulses = []
    vis = torch.from_numpy(synth.generate(wl)).pin_memory()
    h = frbx.Handle.from_workload(wl)
    out = h.search(vis, wl.dms, [1, 2, 4, 8], want_series=True)
    t = h.stage_times()
    assert t["tree_tensor"] == 1 and t["tree_chunks"] <= most
    dev = frbx.Handle.from_workload(wl).search(vis.cuda(), wl.dms, [1, 2, 4, 8], want_series=True)
    assert np.array_equal(out["series"], dev["series"]) and np.array_equal(out["pnorm"], dev["pnorm"])
