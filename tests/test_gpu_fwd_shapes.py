"""Default shapes of forward sweeps of more warps than a multiprocessor holds: the
bits of an explicit one- or two-segment sweep, whatever its threads, for torques and
poses, from joint states and from control points."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name, B", [("R48", 77824), ("R48", 80001), ("R48", 99999),
                                     ("R48", 110001), ("R23", 90003), ("chain32", 80001)])
def test_bits_of_explicit_shapes(name, B):
    from paper_2603_05493_gb300 import _lib, build, wbe
    build()
    desc = {"R48": R.r48, "R23": R.r23, "chain32": lambda: R.deep_chain(32)}[name]()
    rob = wbe.Robot(desc, device=0)
    q, qd, qdd = (torch.from_numpy(v).cuda() for v in I.uniform_states(desc.dof, B, 91))
    T = 64
    U = torch.from_numpy(np.random.default_rng(92).uniform(-1, 1, (B // T, desc.dof, 9))
                         .astype(np.float32)).cuda()
    kw = dict(sphere=False, dmin=False)
    for f in (lambda t: rob.eval(q, qd, qdd, tune=t, **kw),
              lambda t: rob.eval_spline(U, T, 0.1, tune=t, **kw)):
        got = f(None)
        some = [f(wbe.Tune(_lib.WB_KERNEL_TREE, G, 128, 0)) for G in (1, 2)]
        assert all(torch.equal(got["pose"], o["pose"]) for o in some)
        assert any(torch.equal(got["tau"], o["tau"]) for o in some)
        one = f(wbe.Tune(_lib.WB_KERNEL_TREE, 1, 0, 0))
        assert torch.equal(one["tau"], some[0]["tau"])
