"""The eight-lanes-a-configuration pair kernel of small robots: the same bits as
the full map-reduce over every form it accepts -- full and partial pair masks,
no pairs, exact ties, poses far from the origin, not-a-number poses, ragged
batches."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu


def masked(kind):
    desc = R.r7()
    rng = np.random.default_rng(3)
    if kind == "half":
        return desc.with_pairs(desc.pairs[np.sort(rng.permutation(desc.P)[:desc.P // 2])])
    if kind == "one":
        return desc.with_pairs(desc.pairs[100:101])
    if kind == "none":
        return desc.with_pairs(np.zeros((0, 2), np.int32))
    if kind == "ties":  # the spheres of a link coincide: every distance comes 16 times
        from dataclasses import replace
        c, r = desc.sph_c.copy(), desc.sph_r.copy()
        for s in range(desc.S):
            c[s], r[s] = c[4 * (s // 4)], r[4 * (s // 4)]
        return replace(desc, sph_c=c, sph_r=r)
    return desc


def in_index_order(desc, sph):
    """The exact path in numpy: fp32 distances with its operation order (a
    product of fp32 numbers is exact in fp64, so rounding each fused
    multiply-add's fp64 sum to fp32 gives its bits), the least, and of equal
    ones the first pair.  (The full map-reduce's screen bounds its rounding by
    the robot's reach, so it is no reference for poses far beyond that.)"""
    f, d = np.float32, np.float64
    i, j = desc.pairs[:, 0], desc.pairs[:, 1]
    r = desc.sph_r.astype(f)
    x, y, z = ((sph[:, i, k] - sph[:, j, k]).astype(f) for k in range(3))
    s = (x * x).astype(f)
    for v in (y, z):
        s = (v.astype(d) * v.astype(d) + s.astype(d)).astype(f)
    dist = (np.sqrt(s) - (r[i] + r[j])).astype(f)
    if desc.P == 0:
        return np.full(len(sph), np.inf, f), np.full(len(sph), -1)
    return dist.min(1), dist.argmin(1)


@pytest.mark.parametrize("B", [1, 3, 4, 5, 33, 4099])
@pytest.mark.parametrize("kind", ["full", "half", "one", "none", "ties"])
def test_same_bits_as_full_map_reduce(kind, B):
    from paper_2603_05493_gb300 import build, wbe
    build()
    desc = masked(kind)
    rob = wbe.Robot(desc, device=0)
    q = torch.from_numpy(I.uniform_states(desc.dof, B, seed=5)[0]).cuda()
    pose = rob.eval(q, sphere=False, dmin=False, tau=False)["pose"]
    far = pose.clone()
    far[..., 9:] += 300.0
    got = rob.self_collision(pose, diff=True)
    ref = rob.self_collision(pose, diff=True, tune=wbe.TREE_NOCULL)
    for k in ("sphere", "dmin", "worst", "diff"):
        assert torch.equal(got[k], ref[k]), k
    for p in (pose, far):
        got = rob.self_collision(p)
        dmin, worst = in_index_order(desc, got["sphere"].cpu().numpy())
        assert np.array_equal(got["dmin"].cpu().numpy(), dmin)
        assert np.array_equal(got["worst"].cpu().numpy(), worst)
    got = rob.self_collision(pose, sphere=True, dmin=False)
    assert torch.equal(got["sphere"], rob.self_collision(pose)["sphere"])


def test_not_a_number_poses():
    from paper_2603_05493_gb300 import wbe
    desc = R.r7()
    rob = wbe.Robot(desc, device=0)
    q = torch.from_numpy(I.uniform_states(desc.dof, 9, seed=6)[0]).cuda()
    pose = rob.eval(q, sphere=False, dmin=False, tau=False)["pose"]
    ref = rob.self_collision(pose)
    pose[4] = float("nan")
    got = rob.self_collision(pose)
    keep = [b for b in range(9) if b != 4]
    assert torch.equal(got["dmin"][keep], ref["dmin"][keep])
    assert torch.equal(got["worst"][keep], ref["worst"][keep])
    assert got["dmin"][4].item() == float("inf") and got["worst"][4].item() == -1
