"""The largest shift of a DM trial, which the host evaluates for the lowest point: every search and fit checks
its segments against it.  Uneven channel orders, trials whose shifts are exact halves, the largest shifts
an int holds and beyond, against the maximum of the device's own table."""
import numpy as np
import pytest

from tests.test_gpu_tree import frbx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f0", [[1400.0, 1432.0], [3000.0, 10424.0, 5464.0, 2992.0], [32.0, 64.0]])
def test_largest_shift(frbx, f0):  # noqa: F811
    import torch
    h = frbx.Handle(np.array(f0), 4, 16.0, 0.5)
    rng = np.random.default_rng(len(f0))
    dms = np.r_[0.0, 1e-9, rng.uniform(0.0, 3000.0, 200), 1e7, 1e300]
    # trials at the edge between two shifts of the lowest point
    f = (np.array(f0)[:, None] + np.arange(4) * 4.0).reshape(-1)
    per_dm = 4.15e6 * (f.min() ** -2 - f.max() ** -2) / 0.5
    dms = np.r_[dms, (np.arange(1, 60) - 0.5) / per_dm]
    top = h.shift_table(dms).max(axis=1).astype(np.int64)
    T = 200
    vis = torch.zeros((1, T, h.C), dtype=torch.complex64, device="cuda")
    for d in range(len(dms)):
        rows = lambda k0: np.array([[0, d, 1, k0]], np.int32)  # noqa: E731
        last = T - 1 - top[d]
        if last >= 0:
            h.fit_segments(vis, dms, rows(last))
        with pytest.raises(frbx.FrbxError) as e:
            h.fit_segments(vis, dms, rows(max(last + 1, 0)))
        assert e.value.code == frbx.FRBX_EINVAL


def test_no_segments_leaves_nothing_in_flight(frbx):  # noqa: F811
    """A fit of no segments returns once the host cube is read, so the caller may release or rewrite it."""
    import torch
    h = frbx.Handle(np.array([1400.0, 1432.0]), 4, 16.0, 0.5)
    vis = torch.zeros((1, 1 << 22, h.C), dtype=torch.complex64, pin_memory=True)  # 268 MB
    st = torch.cuda.current_stream()
    for _ in range(2):
        assert len(h.fit_segments(vis, np.array([0.0, 50.0]), np.zeros((0, 4), np.int32))) == 0
        assert st.query()
