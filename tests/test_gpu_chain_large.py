"""Batches large enough for the chain kernel (more than 24 warps a multiprocessor),
and just not: the bits of the batched general sweep, whole and with torques alone."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R
from tests.test_gpu_chain import chain

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [116736, 116737, 140001])
@pytest.mark.parametrize("n", [1, 2, 7, 12])
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
    for threads in (64, 128, 256):
        tune = wbe.Tune(kernel=3, lanes_per_config=1, configs_per_block=threads)
        o = rob.eval(q, qd, qdd, sphere=False, dmin=False, tune=tune)
        assert torch.equal(o["pose"], pose) and torch.equal(o["tau"], tau)
        o = rob.eval(q, qd, qdd, pose=False, sphere=False, dmin=False, tune=tune)
        assert torch.equal(o["tau"], tau)
