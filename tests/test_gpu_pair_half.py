"""Block bounds in halves, relative to the first link: the culled pair kernel
(distance, worst pair, bits) and the hinge sum against every pair's fp32
distance, with links anywhere in the robot's reach, the whole
robot moved within it, and one link (the first too) so far away that a half
overflows.  The distances are the kernel's own arithmetic, so they have to be
equal; a hinge term's is within three roundings of 2 m (4e-7), and up to 600
terms a partial sum in fp32 add 600 roundings (4e-5 of the sum)."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu


def distances(desc, sph):
    f, d = np.float32, np.float64
    i, j = desc.pairs[:, 0], desc.pairs[:, 1]
    r = desc.sph_r.astype(f)
    x, y, z = ((sph[:, i, k] - sph[:, j, k]).astype(f) for k in range(3))
    s = (x * x).astype(f)
    for v in (y, z):  # products of fp32 numbers are exact in fp64
        s = (v.astype(d) * v.astype(d) + s.astype(d)).astype(f)
    return (np.sqrt(s) - (r[i] + r[j])).astype(f)


@pytest.mark.parametrize("kind", ["as it is", "moved", "scattered", "first link far", "a link far"])
@pytest.mark.parametrize("robot", ["R48", "R23", "R48 ragged"])
def test_bounds(robot, kind):
    from paper_2603_05493_gb300 import build, wbe
    build()
    desc = R.r23() if robot == "R23" else R.r48()
    rng = np.random.default_rng(11)
    if robot == "R48 ragged":
        desc = desc.with_pairs(desc.pairs[np.sort(rng.permutation(desc.P)[:desc.P // 5])])
    rob = wbe.Robot(desc, device=0)
    B = 37
    q = torch.from_numpy(I.uniform_states(desc.dof, B, seed=12)[0]).cuda()
    pose = rob.eval(q, sphere=False, dmin=False, tau=False)["pose"]
    n = pose.shape[-2]
    if kind == "moved":
        pose[..., 9:] += 0.25
    elif kind == "scattered":
        pose[..., 9:] += torch.from_numpy(rng.uniform(-0.3, 0.3, (B, n, 3)).astype(np.float32)).cuda()
    elif kind == "first link far":
        pose[:, 0, 9:] += 1e5
    elif kind == "a link far":
        pose[:, n // 2, 9:] -= 1e5
    got = rob.self_collision(pose, bits=True)
    dist = distances(desc, got["sphere"].cpu().numpy())
    assert np.array_equal(got["dmin"].cpu().numpy(), dist.min(1))
    assert np.array_equal(got["worst"].cpu().numpy(), dist.argmin(1))
    words = got["bits"].cpu().numpy().view(np.uint32)
    on = (words[:, np.arange(desc.P) // 32] >> (np.arange(desc.P) % 32).astype(np.uint32)) & 1
    assert np.array_equal(on.astype(bool), dist < 0)
    eta = 0.05
    cost, _ = rob.self_collision_hinge(pose, eta, 1.0)
    terms = np.maximum(0.0, eta - dist.astype(np.float64))
    tol = 4e-7 * (terms > 0).sum(1) + 4e-5 * terms.sum(1) + 1e-7
    assert np.all(np.abs(cost.cpu().numpy() - terms.sum(1)) <= tol)
