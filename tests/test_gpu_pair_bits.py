"""Colliding-pair bits of the culled pair kernel, decided on squared distances
with the square root only near touching: every bit against the exact fp32
distance, for full and partial blocks, ragged last words, and spheres that
touch exactly or miss by an ulp."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from synthetic import inputs as I
from synthetic import robots as R

pytestmark = pytest.mark.gpu


def exact_bits(desc, sph):
    """sqrt(|c_i - c_j|^2) - (r_i + r_j) < 0 in fp32 with fused multiply-adds
    (products of fp32 numbers are exact in fp64)."""
    f, d = np.float32, np.float64
    i, j = desc.pairs[:, 0], desc.pairs[:, 1]
    r = desc.sph_r.astype(f)
    x, y, z = ((sph[:, i, k] - sph[:, j, k]).astype(f) for k in range(3))
    s = (x * x).astype(f)
    for v in (y, z):
        s = (v.astype(d) * v.astype(d) + s.astype(d)).astype(f)
    return np.sqrt(s) - (r[i] + r[j]) < 0


@pytest.mark.parametrize("B", [1, 5, 70])
@pytest.mark.parametrize("kind", ["R48", "R23", "R48 partial", "R48 touching"])
def test_bits(kind, B):
    from paper_2603_05493_gb300 import build, wbe
    build()
    desc = R.r23() if kind == "R23" else R.r48()
    rng = np.random.default_rng(B)
    if kind == "R48 partial":
        desc = desc.with_pairs(desc.pairs[np.sort(rng.permutation(desc.P)[:desc.P // 3])])
    q = torch.from_numpy(I.uniform_states(desc.dof, B, seed=B)[0]).cuda()
    if kind == "R48 touching":
        # radii so that many pairs of the first configuration touch to an ulp
        rob = wbe.Robot(desc, device=0)
        c = rob.eval(q[:, :1].contiguous(), tau=False)["sphere"][0].cpu().numpy()
        r = desc.sph_r.astype(np.float32)
        for p in range(0, desc.P, 97):
            i, j = desc.pairs[p]
            gap = np.float32(np.linalg.norm((c[i] - c[j]).astype(np.float64))) - r[i]
            if 0.01 < gap < 0.5:
                r[j] = gap
        desc = replace(desc, sph_r=r.astype(np.float64))
    rob = wbe.Robot(desc, device=0)
    o = rob.eval(q, tau=False, bits=True)
    words = o["bits"].cpu().numpy().view(np.uint32)
    got = (words[:, np.arange(desc.P) // 32] >> (np.arange(desc.P) % 32).astype(np.uint32)) & 1
    assert np.array_equal(got.astype(bool), exact_bits(desc, o["sphere"].cpu().numpy()))
