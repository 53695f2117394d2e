"""Spline forward sweeps asked for at the edge of a block's shared memory: robots
whose 8-segment plan shares so many links that the partials of 512 threads, the
link records and the basis rows together pass the limit by a few kilobytes.  The
call runs with fewer threads and gives the same bits."""
import numpy as np
import pytest
import torch

from synthetic import robots as R

pytestmark = pytest.mark.gpu


def brooms(handles):
    """255 links: four handles of the given lengths, each with a brush of single
    links on its last one; an 8-segment plan cuts every brush and shares its
    handle."""
    parent = []
    for length, links in zip(handles, (64, 64, 64, 63)):
        for i in range(links):
            parent.append(-1 if i == 0 else top if i > length else len(parent) - 1)
            if i == length - 1:
                top = len(parent) - 1
    n = len(parent)
    rng = np.random.default_rng(3)
    axis = rng.normal(size=(n, 3))
    return R._plain("brooms", parent, [R.REVOLUTE] * n, axis / np.linalg.norm(axis, axis=1)[:, None],
                    [R._Tp(*rng.uniform(-0.1, 0.1, 3)) for _ in range(n)], mass=rng.uniform(0.5, 1, n),
                    com=rng.uniform(-0.1, 0.1, (n, 3)), Icom=[[0.1, 0.1, 0.1, 0, 0, 0]] * n,
                    sph_link=[0], sph_c=np.zeros((1, 3)), sph_r=[0.1])


@pytest.mark.parametrize("handles", [(20, 20, 20, 20), (21, 21, 21, 22), (21, 21, 22, 22),
                                     (21, 22, 22, 22)])
def test_same_bits_with_fewer_threads(handles):
    from paper_2603_05493_gb300 import _lib, build, wbe
    build()
    desc = brooms(handles)
    rob = wbe.Robot(desc, device=0)
    U = torch.from_numpy(np.random.default_rng(4).uniform(-1, 1, (3, desc.dof, 7)).astype(np.float32))
    U = U.cuda()
    got, ref = (rob.eval_spline(U, 50, 0.1, sphere=False, dmin=False,
                                tune=wbe.Tune(_lib.WB_KERNEL_TREE, 8, threads, 0))
                for threads in (512, 256))
    torch.cuda.synchronize()
    assert torch.equal(got["tau"], ref["tau"]) and torch.equal(got["pose"], ref["pose"])
    assert torch.isfinite(got["tau"]).all()
