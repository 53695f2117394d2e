"""Which kinematics kernel a call takes goes by its batch and its outputs; both give
the same bits: every batch equal to the same configurations in small and in large
batches, for each count of outputs that the rule knows."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("com", [False, True])
@pytest.mark.parametrize("targets", [[], [4], [0], [6, 2], [1, 3, 6]])
@pytest.mark.parametrize("name", ["R7", "R23"])
def test_batches_agree(name, targets, com):
    from paper_2603_05493_gb300 import build, wbe
    build()
    if not targets and not com:
        pytest.skip("nothing asked for")
    desc = R.r7() if name == "R7" else R.r23()
    rob = wbe.Robot(desc, device=0)
    B = 40000
    q = torch.from_numpy(I.uniform_states(desc.dof, B, seed=41)[0]).cuda()
    pose = rob.eval(q, sphere=False, dmin=False, tau=False)["pose"]

    def call(lo, hi):
        return [x for x in rob.kinematics(pose[lo:hi].contiguous(), targets, com=com, jac_com=com)
                if x is not None]

    whole = call(0, B)
    assert all(torch.isfinite(x).all() for x in whole)
    for lo, hi in ((0, 1), (1, 258), (300, 12345), (12345, B)):
        for a, b in zip(call(lo, hi), whole):
            assert torch.equal(a, b[lo:hi])
