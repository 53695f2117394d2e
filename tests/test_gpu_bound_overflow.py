"""Block bounds in halves where a coordinate difference overflows one: two links
at -4e4 and 4e4 from the first.  Their block has to be kept -- it holds the
active pairs of a summed hinge, or with large radii the closest pair.

Reference: every pair's distance from the kernel's own fp32 centres, in its own
arithmetic for the minimum and the bits, and in fp64 for the sum (a term within 8
roundings of its parts, each of at most `adds` additions a lane within 2^-24 of
the sum)."""
import numpy as np
import pytest
import torch

from synthetic import robots as R
from tests.test_gpu_pair_half import distances

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


def apart(per, radius, step, ragged):
    """Eleven links on a root: the first two 8e4 apart with `per` spheres of the
    given radius each, the others in a row, `step` apart; masked in are the pairs of
    those two and the neighbours' among the rest."""
    rng = np.random.default_rng(9)
    n = 12
    at = [(0, 0, 0), (-4e4, 0, 0), (4e4, 0, 0)] + [(0, step * k, 0) for k in range(9)]
    link = np.repeat(np.arange(1, n), per)
    r = np.where(link < 3, radius, 0.5)
    pairs = [(a, b) for a in range(len(link)) for b in range(a + 1, len(link))
             if (link[a], link[b]) == (1, 2) or (link[a] > 2 and link[b] == link[a] + 1)]
    if ragged:
        pairs = [p for k, p in enumerate(pairs) if k % 5]
    return R._plain("apart", [-1] + [0] * (n - 1), [R.REVOLUTE] * n, [[0, 0, 1]] * n,
                    [R._Tp(*p) for p in at], mass=[1.0] * n, com=np.zeros((n, 3)),
                    Icom=[[0.1, 0.1, 0.1, 0, 0, 0]] * n, sph_link=link,
                    sph_c=rng.uniform(-0.4, 0.4, (len(link), 3)), sph_r=r, pairs=pairs)


@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("per", [4, 3])
@pytest.mark.parametrize("radius, step", [(0.5, 3.0), (3.2e4, 3e4), (5e4, 3.0)])
def test_kept(per, radius, step, ragged):
    from paper_2603_05493_gb300 import build, wbe
    build()
    desc = apart(per, radius, step, ragged)
    rob = wbe.Robot(desc, device=0)
    q = torch.zeros((desc.dof, 3), device="cuda")
    q[1:, 1] = 0.7
    pose = rob.eval(q, sphere=False, dmin=False, tau=False)["pose"]
    got = rob.self_collision(pose, bits=True)
    sph = got["sphere"].cpu().numpy()
    dist = distances(desc, sph)
    assert np.array_equal(got["dmin"].cpu().numpy(), dist.min(1))
    assert np.array_equal(got["worst"].cpu().numpy(), dist.argmin(1))
    words = got["bits"].cpu().numpy().view(np.uint32)
    on = (words[:, np.arange(desc.P) // 32] >> (np.arange(desc.P) % 32).astype(np.uint32)) & 1
    assert np.array_equal(on.astype(bool), dist < 0)
    eta = 9e4
    cost, _ = rob.self_collision_hinge(pose, eta, 1.0)
    i, j = desc.pairs[:, 0], desc.pairs[:, 1]
    nrm = np.linalg.norm(sph.astype(np.float64)[:, i] - sph.astype(np.float64)[:, j], axis=-1)
    rs = desc.sph_r[i] + desc.sph_r[j]
    term = np.maximum(0.0, eta - (nrm - rs))
    adds = 16 * (-(-desc.P // 32) + 1) + 8  # blocks are at most the pairs
    tol = (8 * EPS * (nrm + eta + rs)).sum(1) + adds * EPS * term.sum(1)
    assert np.all(np.abs(cost.cpu().numpy() - term.sum(1)) <= tol)
