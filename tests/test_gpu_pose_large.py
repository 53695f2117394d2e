"""Poses alone of batches beyond the L2, where the sweeps' blocks are limited: the bits
of small batches, from joint states and from control points, at the limit's edges."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name, B", [("R48", 80003), ("R48", 97281), ("R48", 131073),
                                     ("R23", 106400), ("R7", 350001)])
def test_bits_of_small_batches(name, B):
    from paper_2603_05493_gb300 import build, wbe
    build()
    desc = {"R48": R.r48, "R23": R.r23, "R7": R.r7}[name]()
    rob = wbe.Robot(desc, device=0)
    q = torch.from_numpy(I.uniform_states(desc.dof, B, seed=61)[0]).cuda()
    kw = dict(sphere=False, dmin=False, tau=False)
    pose = rob.eval(q, **kw)["pose"]
    for lo, hi in ((0, 700), (B // 2, B // 2 + 999), (B - 33, B)):
        assert torch.equal(rob.eval(q[:, lo:hi].contiguous(), **kw)["pose"], pose[lo:hi])
    T = 64
    U = torch.from_numpy(np.random.default_rng(62).uniform(-1, 1, (B // T, desc.dof, 9))
                         .astype(np.float32)).cuda()
    pose = rob.eval_spline(U, T, 0.1, **kw)["pose"]
    for lo, hi in ((0, 5), (B // T - 3, B // T)):
        got = rob.eval_spline(U[lo:hi].clone(), T, 0.1, **kw)["pose"]
        assert torch.equal(got, pose[lo * T:hi * T])
