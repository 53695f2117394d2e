"""The autograd node with outputs left out of the loss: an output without a gradient
reaches the kernels as none, for every subset of the outputs and every kernel
family; against the same call given explicit zeros (the largest difference within
1e-5 of the largest gradient: the instances that leave a gradient out add no zeros)."""
import itertools

import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu

OUTS = ("pose", "sphere", "dmin", "tau")
SUBSETS = [s for n in (1, 2, 3) for s in itertools.combinations(OUTS, n)]


@pytest.mark.parametrize("kname", ["default", "fused", "plain"])
@pytest.mark.parametrize("name", ["R23", "mixed"])
def test_subsets(name, kname):
    from paper_2603_05493_gb300 import build, wbe
    build()
    desc = R.r23() if name == "R23" else R.mixed_joint_tree()
    rob = wbe.Robot(desc, device=0)
    tune = {"default": None, "fused": wbe.FUSED, "plain": wbe.PLAIN}[kname]
    B = 41
    x = [torch.from_numpy(np.ascontiguousarray(v, dtype=np.float32)).cuda()
         for v in I.uniform_states(desc.dof, B, 81)]
    g = dict(zip(OUTS, (torch.from_numpy(v).cuda() for v in I.upstream_grads(desc, B, 82))))
    for on in SUBSETS:
        leaf = [v.clone().requires_grad_(True) for v in x]
        out = dict(zip(OUTS, wbe.whole_body_eval(rob, *leaf, tune=tune)[:4]))
        sum((out[k] * g[k]).sum() for k in on).backward()
        ref_leaf = [v.clone().requires_grad_(True) for v in x]
        ref = dict(zip(OUTS, wbe.whole_body_eval(rob, *ref_leaf, tune=tune)[:4]))
        torch.autograd.backward([ref[k] for k in OUTS],
                                [g[k] if k in on else torch.zeros_like(g[k]) for k in OUTS])
        for a, b in zip(leaf, ref_leaf):
            assert (a.grad - b.grad).abs().max() <= 1e-5 * b.grad.abs().max() + 1e-7, on
