"""Small robots' pair stage: which of two kernels a call takes goes by its batch,
spheres and pairs; both give the same bits.  Every batch against its pieces, for
robots on both sides of the rule and batches around its crossings."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu


def robot(links, pairs):
    desc = R._build("s", 5 + links, list(range(-1, links - 1)), [R.REVOLUTE] * links, 0, 0.03, 0.08,
                    2 if links > 2 else 1)
    if pairs and pairs < desc.P:
        keep = np.random.default_rng(links).permutation(desc.P)[:pairs]
        desc = desc.with_pairs(desc.pairs[np.sort(keep)])
    return desc


@pytest.mark.parametrize("links, pairs", [(2, 0), (3, 0), (4, 16), (7, 1), (7, 16), (7, 0), (8, 100)])
def test_batches_agree(links, pairs):
    from paper_2603_05493_gb300 import build, wbe
    build()
    desc = robot(links, pairs)
    rob = wbe.Robot(desc, device=0)
    B = 131073
    q = torch.from_numpy(I.uniform_states(desc.dof, B, seed=71)[0]).cuda()
    pose = rob.eval(q, sphere=False, dmin=False, tau=False)["pose"]
    small = [rob.self_collision(pose[lo:lo + 8192].contiguous(), diff=True)
             for lo in range(0, B, 8192)]
    ref = {k: torch.cat([o[k] for o in small]) for k in ("sphere", "dmin", "worst", "diff")}
    for n in (16383, 20011, 32768, 50001, 99999, B):
        got = rob.self_collision(pose[:n].contiguous(), diff=True)
        for k in ref:
            assert torch.equal(got[k], ref[k][:n]), (k, n)
