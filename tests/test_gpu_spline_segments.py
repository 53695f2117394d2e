"""Default shapes of the forward sweep from control points: the segments of the sweep
of joint states at every batch size, so that poses and torques are the same bits."""
import numpy as np
import pytest
import torch

from synthetic import robots as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["R48", "R23", "R7"])
@pytest.mark.parametrize("n_traj", [80, 313, 1215, 1217, 1250, 1562, 1719, 2048])
def test_equal_to_the_two_step_path(name, n_traj):
    from paper_2603_05493_gb300 import build, wbe
    build()
    desc = {"R48": R.r48, "R23": R.r23, "R7": R.r7}[name]()
    rob = wbe.Robot(desc, device=0)
    T = 64
    U = torch.from_numpy(np.random.default_rng(92).uniform(-1, 1, (n_traj, desc.dof, 9))
                         .astype(np.float32)).cuda()
    kw = dict(sphere=False, dmin=False)
    a = rob.eval(*wbe.bspline_eval(U, T, 0.1), **kw)
    b = rob.eval_spline(U, T, 0.1, **kw)
    assert torch.equal(a["pose"], b["pose"])
    assert torch.equal(a["tau"], b["tau"])
