"""The forward sweep of robots without branches: the same bits as the general
one-segment sweep (which a batch of one problem runs), over chain lengths, joint
types with fixed links between, ragged batches and block sizes."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu


def chain(n):
    kinds = [R.REVOLUTE, R.PRISMATIC, R.REVOLUTE, R.FIXED, R.REVOLUTE]
    jt = [kinds[k % 5] if n > 1 else R.REVOLUTE for k in range(n)]
    return R._build("chain%d" % n, 90 + n, [k - 1 for k in range(n)], jt, 1, 0.03, 0.08, 2)


@pytest.mark.parametrize("B", [1, 33, 1000])
@pytest.mark.parametrize("n", [1, 2, 7, 20, 31])
def test_same_bits_as_the_general_sweep(n, B):
    from paper_2603_05493_gb300 import build, wbe
    build()
    desc = R.r7() if n == 7 else chain(n)
    rob = wbe.Robot(desc, device=0)
    q, qd, qdd = (torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()
                  for x in I.uniform_states(desc.dof, B, seed=n))
    batch = wbe.Batch([rob], [(0, B)])
    batch.set_tune(fwd_segments=[1], bwd_segments=[1])
    pose = torch.empty((B, desc.n, 12), device="cuda")
    tau = torch.empty((desc.dof, B), device="cuda")
    batch.eval(q, qd, qdd, pose, tau=tau)
    for threads in (32, 64, 128, 256):
        o = rob.eval(q, qd, qdd, sphere=False, dmin=False,
                     tune=wbe.Tune(kernel=3, lanes_per_config=1, configs_per_block=threads))
        assert torch.equal(o["pose"], pose) and torch.equal(o["tau"], tau)
        o = rob.eval(q, qd, qdd, pose=False, sphere=False, dmin=False,
                     tune=wbe.Tune(kernel=3, lanes_per_config=1, configs_per_block=threads))
        assert torch.equal(o["tau"], tau)
