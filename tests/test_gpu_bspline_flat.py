"""The control-point gradient where its deal changes: more knots than samples, few
rows and many, rows at 256 knots, one and two samples a row; the same check and
tolerance as for the other shapes."""
import pytest

from tests.test_gpu_bspline_rows import test_knot_gradient as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ends", [False, True])
@pytest.mark.parametrize("n_traj,d,K,T", [
    (1, 3, 257, 300), (2, 3, 256, 284), (1, 2, 600, 1100), (3, 2, 900, 40), (450, 1, 256, 40),
    (450, 1, 257, 40), (1, 3, 1024, 1100), (300, 2, 4, 2), (70, 3, 5, 17), (399, 1, 18, 20),
    (401, 1, 18, 20), (401, 1, 30, 20), (401, 1, 29, 20)])
def test_deals(n_traj, d, K, T, ends):
    check(n_traj, d, K, T, ends)
