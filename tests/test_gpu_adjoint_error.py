"""The backward sweep's error against the FP64 oracle, over every robot, its
sweep segments and ragged sizes.  Each link is visited twice (push and close)
and each visit rounds the carried vectors a few times; 4 ulp a visit over the
2 n visits of the longest carried state bounds the relative error of the whole
gradient by 8 n x 6e-8."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu

ROBOTS = {"R7": R.r7, "R23": R.r23, "R48": R.r48, "mixed": R.mixed_joint_tree}


@pytest.mark.parametrize("name", sorted(ROBOTS))
@pytest.mark.parametrize("segments,B", [(1, 1), (1, 95), (2, 33), (4, 64), (8, 65)])
def test_gradient_error(name, segments, B):
    from oracle import oracle as O
    from paper_2603_05493_gb300 import build, wbe
    build()
    O.build()
    desc = ROBOTS[name]()
    rob = wbe.Robot(desc, device=0)
    q, qd, qdd = I.uniform_states(desc.dof, B, seed=70 + B)
    gp, gs, _, gt = I.upstream_grads(desc, B, seed=80 + B)
    ref = O.gradient(desc, q, qd, qdd, gp, gs, None, gt)
    cu = lambda x: torch.from_numpy(x).cuda()  # noqa: E731
    tune = wbe.Tune(kernel=wbe.L.WB_KERNEL_TREE, lanes_per_config=segments)
    try:
        got = rob.eval_backward(cu(q), cu(qd), cu(qdd), None, cu(gp), cu(gs), None, cu(gt),
                                tune=tune)
    except wbe.L.WbError as e:  # a joint driving several links, or fewer links than segments
        assert segments > 1 and "segment" in str(e)
        return
    for g, r in zip(got, ref):
        err = np.linalg.norm(g.cpu().numpy() - r) / np.linalg.norm(r)
        assert err <= 8 * desc.n * 6e-8
