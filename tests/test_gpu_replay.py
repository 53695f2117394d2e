"""Segmented forward sweeps of the deepest chains and trees, whose segments replay up
to 31 ancestors: the poses have the bits of the one-segment sweep (the replay is the
same arithmetic), the torques are within the summation order of the shared links'
partials (1e-5 of the largest), single and batched."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["chain32", "max255", "R48"])
def test_poses_and_torques(name):
    from paper_2603_05493_gb300 import _lib, build, wbe
    build()
    desc = {"chain32": lambda: R.deep_chain(32), "max255": R.max_size, "R48": R.r48}[name]()
    rob = wbe.Robot(desc, device=0)
    B = 67
    x = I.uniform_states(desc.dof, B, seed=51)
    q, qd, qdd = (torch.from_numpy(v).cuda() for v in x)

    def call(G, tau=True):
        return rob.eval(q, qd, qdd, sphere=False, dmin=False, tau=tau,
                        tune=wbe.Tune(_lib.WB_KERNEL_TREE, G, 0, 0))

    ref = call(1)
    scale = ref["tau"].abs().max(0).values
    for G in (2, 4, 8):
        got = call(G)
        assert torch.equal(got["pose"], ref["pose"])
        assert torch.equal(call(G, tau=False)["pose"], ref["pose"])
        assert ((got["tau"] - ref["tau"]).abs() <= 1e-5 * scale).all()
    batch = wbe.Batch([rob], [(0, 33), (0, 34)])
    st = [torch.cat([v[:, :33].reshape(-1), v[:, 33:].reshape(-1)]) for v in (q, qd, qdd)]
    pose, tau = batch.empty("pose"), batch.empty("joint")
    batch.eval(*st, pose, None, None, None, tau)
    assert torch.equal(pose.reshape(ref["pose"].shape), ref["pose"])
    got = torch.cat([tau[:33 * desc.dof].reshape(-1, 33), tau[33 * desc.dof:].reshape(-1, 34)], 1)
    assert ((got - ref["tau"]).abs() <= 1e-5 * scale).all()
