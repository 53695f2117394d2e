"""The kernel that bench.py names for the arm's forward sweep is the one that runs."""
import numpy as np
import pytest
import torch

import bench
from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B, seg", [(131072, 1), (116736, 1), (4096, 1), (4096, 2)])
def test_arm_sweep(B, seg):
    from torch.profiler import ProfilerActivity, profile

    from paper_2603_05493_gb300 import _lib, build, wbe
    build()
    desc = R.r7()
    rob = wbe.Robot(desc, device=0)
    x = [torch.from_numpy(np.ascontiguousarray(v, dtype=np.float32)).cuda()
         for v in I.uniform_states(desc.dof, B, 1)]
    tune = wbe.Tune(_lib.WB_KERNEL_TREE, seg, 0, 0)
    names = []
    for _ in range(2):  # the profiler's first range can come back empty
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            rob.eval(*x, sphere=False, dmin=False, tune=tune)
            torch.cuda.synchronize()
        names = [e.key for e in p.key_averages() if "tree_fwd" in e.key]
    if not names:
        pytest.skip("the profiler sees no kernels here")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert any(bench.arm_sweep_kernel(seg, B, sms) in n for n in names), names
