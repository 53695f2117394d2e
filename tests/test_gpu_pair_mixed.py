"""The culled pair stage and the summed hinge of robots whose groups of 4 spheres
lie over several links (1, 3 or 5 spheres a link; the last group partly filled)
beside ones that do not, with every pair of different links masked in or three in
five of them, and with so many blocks that their bounds are not kept: the
distance, the worst pair and the bits equal to every pair's fp32 distance, the sum
to its terms in fp64 (a term within 8 roundings of its parts, at most `adds`
additions a lane)."""
import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R
from tests.test_gpu_pair_half import distances

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


def star(links, per, ragged):
    """`links` three-link legs from a root, `per` spheres a link."""
    rng = np.random.default_rng(links + per)
    n = links + 1
    parent = [-1] + [0 if k % 3 == 0 else k for k in range(links)]
    link = np.repeat(np.arange(1, n), per)
    i, j = np.triu_indices(len(link), 1)
    on = link[i] != link[j]
    if ragged:
        on &= rng.random(len(i)) < 0.6
    axis = rng.normal(size=(n, 3))
    return R._plain("star", parent, [R.REVOLUTE] * n, axis / np.linalg.norm(axis, axis=1)[:, None],
                    [R._Tp(*rng.uniform(-0.4, 0.4, 3)) for _ in range(n)], mass=[1.0] * n,
                    com=np.zeros((n, 3)), Icom=[[0.1, 0.1, 0.1, 0, 0, 0]] * n, sph_link=link,
                    sph_c=rng.uniform(-0.1, 0.1, (len(link), 3)),
                    sph_r=rng.uniform(0.01, 0.05, len(link)), pairs=np.stack([i[on], j[on]], 1))


@pytest.mark.parametrize("crowded", [False, True])
@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("links, per", [(11, 3), (33, 1), (12, 4), (9, 5), (60, 4), (81, 3)])
def test_against_every_pair(links, per, ragged, crowded):
    from paper_2603_05493_gb300 import build, wbe
    build()
    desc = star(links, per, ragged)
    rob = wbe.Robot(desc, device=0)
    q = torch.from_numpy(I.uniform_states(desc.dof, 21, seed=31)[0]).cuda()
    pose = rob.eval(q, sphere=False, dmin=False, tau=False)["pose"]
    if crowded:  # the links drawn together, so that many pairs collide
        pose[..., 9:] *= 0.15
    got = rob.self_collision(pose, bits=True)
    sph = got["sphere"].cpu().numpy()
    dist = distances(desc, sph)
    assert np.array_equal(got["dmin"].cpu().numpy(), dist.min(1))
    assert np.array_equal(got["worst"].cpu().numpy(), dist.argmin(1))
    words = got["bits"].cpu().numpy().view(np.uint32)
    on = (words[:, np.arange(desc.P) // 32] >> (np.arange(desc.P) % 32).astype(np.uint32)) & 1
    assert np.array_equal(on.astype(bool), dist < 0)
    if crowded:
        assert 0.005 < on.mean() < 0.5
    alone = rob.self_collision(pose)
    assert torch.equal(alone["dmin"], got["dmin"]) and torch.equal(alone["worst"], got["worst"])
    eta = 0.05
    cost, _ = rob.self_collision_hinge(pose, eta, 1.0)
    i, j = desc.pairs[:, 0], desc.pairs[:, 1]
    nrm = np.linalg.norm(sph.astype(np.float64)[:, i] - sph.astype(np.float64)[:, j], axis=-1)
    rs = desc.sph_r[i] + desc.sph_r[j]
    term = np.maximum(0.0, eta - (nrm - rs))
    adds = 16 * (-(-desc.P // 32) + 1) + 8  # blocks are at most the pairs
    tol = (8 * EPS * (nrm + eta + rs)).sum(1) + adds * EPS * term.sum(1)
    assert np.all(np.abs(cost.cpu().numpy() - term.sum(1)) <= tol)
