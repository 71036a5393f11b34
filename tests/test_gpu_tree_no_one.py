"""Window sets without one-AP windows take an instance of the tensor-core window tree that forms no
AP's own maximum: every segment against the FP64 oracle, for blocks of 32 and of 48 columns, on the whole
grid and with an MBD window."""
import pytest

from tests.test_gpu_tree import frbx  # noqa: F401
from tests.test_gpu_tree_cols import _check, _wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("windows", [[2], [4, 2], [8], [2, 64]])
@pytest.mark.parametrize("lm", [64, 256])
def test_no_one_ap_window(frbx, lm, windows):  # noqa: F811
    _check(frbx, _wl(lm, 150, windows))
    cell = 1000.0 / (lm * 16.0)
    _check(frbx, _wl(lm, 150, windows), (5 * cell, 20 * cell))
