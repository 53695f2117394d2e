"""The one-link-per-joint kinematics kernel: sliding joints and mimic factors,
target lists past 32, one configuration and ragged passes, against the oracle
with the tolerances of the kinematics tests (2e-5 per unit rate, 1e-5 m)."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu


def sliding():
    desc = R.r23()
    jtype, mult, off = desc.jtype.copy(), desc.mimic_mult.copy(), desc.mimic_off.copy()
    jtype[[3, 8, 20]] = R.PRISMATIC
    mult[5], off[5] = -0.5, 0.25
    return replace(desc, jtype=jtype, mimic_mult=mult, mimic_off=off)


@pytest.mark.parametrize("B,nt", [(1, 1), (9, 0), (33, 40), (4097, 2), (5, 64)])
def test_against_oracle(B, nt):
    from oracle import oracle as O
    from paper_2603_05493_gb300 import build, wbe
    build()
    O.build()
    desc = sliding()
    rob = wbe.Robot(desc, device=0)
    q = I.uniform_states(desc.dof, B, seed=B)[0]
    q[[2, 7, 19]] *= 0.1  # sliding joints within 0.3 m
    pose = rob.eval(torch.from_numpy(q).cuda(), sphere=False, dmin=False, tau=False)["pose"]
    targets = [(7 * t + 3) % desc.n for t in range(nt)]
    jac, com, jac_com = rob.kinematics(pose, targets)
    idx = np.unique(np.linspace(0, B - 1, 9).astype(int))
    rJ, rcom, rJc = O.kinematics(desc, np.ascontiguousarray(q[:, idx]), targets or [0])
    if nt:
        assert np.abs(jac.cpu().numpy()[idx] - rJ).max() <= 2e-5
        assert (jac.cpu().numpy()[idx][rJ == 0.0] == 0.0).all()
    assert np.abs(com.cpu().numpy()[idx] - rcom).max() <= 1e-5
    assert np.abs(jac_com.cpu().numpy()[idx] - rJc).max() <= 2e-5
