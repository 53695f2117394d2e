"""The summed hinge where the schedule's null entries pass the block bounds: an
activation distance beyond the null entries' far sphere, and a first group of
spheres so far from the first link that its bound is no number.  Every masked
pair counts once and nothing else does.

Reference: the kernel's own fp32 centres, distances and sums in fp64.  A
term eta - d is within 8 roundings of its parts (the centre distance, eta and the
radii, below 1 m); a cost adds its lanes'
terms one after the other (at most 16 for each 32 blocks, and 5 across the
lanes), each add within 2^-24 of the sum so far; a sphere's gradient is a sum of
one unit vector a pair (8 roundings each)."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


def check(desc, rob, pose, eta, w):
    sph = rob.self_collision(pose)["sphere"].cpu().numpy().astype(np.float64)
    cost, g = (t.cpu().numpy().astype(np.float64) for t in rob.self_collision_hinge(pose, eta, w))
    i, j = desc.pairs[:, 0], desc.pairs[:, 1]
    diff = sph[:, i] - sph[:, j]
    nrm = np.linalg.norm(diff, axis=-1)
    term = np.maximum(0.0, eta - (nrm - desc.sph_r[i] - desc.sph_r[j]))
    ref = w * term.sum(1)
    adds = 16 * (-(-len(desc.pairs) // (16 * 32)) + 1) + 8
    tol = w * (8 * EPS * (nrm + eta + 1.0) * (term > 0)).sum(1) + adds * EPS * ref
    assert np.all(np.abs(cost - ref) <= tol), (cost - ref, tol)
    unit = np.where(nrm > 0, 1.0 / np.maximum(nrm, 1e-300), 0.0)[..., None] * diff * (term > 0)[..., None]
    ref_g = np.zeros_like(sph)
    count = np.zeros(sph.shape[:2])
    for p in range(desc.P):
        ref_g[:, i[p]] -= w * unit[:, p]
        ref_g[:, j[p]] += w * unit[:, p]
        count[:, i[p]] += term[:, p] > 0
        count[:, j[p]] += term[:, p] > 0
    tol_g = w * EPS * count * (count + 8) + 1e-12
    assert np.all(np.abs(g - ref_g).max(-1) <= tol_g)


@pytest.fixture(scope="module")
def W():
    from paper_2603_05493_gb300 import build, wbe
    build()
    return wbe


@pytest.mark.parametrize("eta", [1e5, 1.5e5, 1e6])
@pytest.mark.parametrize("name", ["R7", "R48", "R7 half"])
def test_activation_beyond_the_far_sphere(W, name, eta):
    desc = R.r48() if name == "R48" else R.r7()
    if name == "R7 half":
        desc = desc.with_pairs(desc.pairs[::2])
    rob = W.Robot(desc, device=0)
    q = torch.from_numpy(I.uniform_states(desc.dof, 9, seed=21)[0]).cuda()
    check(desc, rob, rob.eval(q, tau=False)["pose"], eta, 0.75)


def fan(groups):
    """A root link without spheres and `groups` links on it with a run of 4
    spheres each, every pair of spheres of different links masked in."""
    n = groups + 1
    rng = np.random.default_rng(5)
    sph_link = np.repeat(np.arange(1, n), 4)
    pairs = [[a, b] for a in range(4 * groups) for b in range(a + 1, 4 * groups) if a // 4 != b // 4]
    return R._plain("fan", [-1] + [0] * groups, [R.REVOLUTE] * n, [[0, 0, 1]] * n,
                    [R._Tp(*rng.uniform(-0.3, 0.3, 3)) for _ in range(n)], mass=[1.0] * n,
                    com=np.zeros((n, 3)), Icom=[[0.1, 0.1, 0.1, 0, 0, 0]] * n, sph_link=sph_link,
                    sph_c=rng.uniform(-0.1, 0.1, (4 * groups, 3)),
                    sph_r=rng.uniform(0.02, 0.05, 4 * groups), pairs=pairs)


@pytest.mark.parametrize("kind", ["far", "not finite"])
@pytest.mark.parametrize("groups", [3, 11])
def test_first_link_away_from_the_spheres(W, groups, kind):
    desc = fan(groups)
    rob = W.Robot(desc, device=0)
    q = torch.from_numpy(I.uniform_states(desc.dof, 7, seed=22)[0]).cuda()
    pose = rob.eval(q, tau=False)["pose"]
    pose[:, 0, 9:] = float("inf") if kind == "not finite" else 1e5  # no sphere sits on it
    check(desc, rob, pose, 0.05, 1.25)
