"""The control-point gradient's blocks of trajectories: staged rows and rows too
long to stage, one and several trajectories a block, ragged last blocks, with
and without boundary conditions and the added gradients, against the adjoint of
the forward in fp64 (the sum of a knot over its samples: at most 4 T / (K - 3)
+ 4 fp32 terms, bounded by that many half-ulps of the largest partial sum)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def rows(wbe, K, T, dt):
    """The forward's own basis rows [3][T][K], probed with unit control points."""
    U = torch.eye(K, device="cuda").reshape(K, 1, K).contiguous()
    return [x.reshape(K, T).T.double().cpu().numpy() for x in wbe.bspline_eval(U, T, dt)]


@pytest.mark.parametrize("ends", [False, True])
@pytest.mark.parametrize("n_traj,d,K,T", [(1, 1, 4, 2), (33, 3, 16, 64), (300, 2, 5, 17),
                                          (3, 2, 300, 40), (2, 2, 7, 1100), (5, 2, 6, 700)])
def test_knot_gradient(n_traj, d, K, T, ends):
    from paper_2603_05493_gb300 import build, wbe
    build()
    rng = np.random.default_rng(T + K)
    g = [rng.standard_normal((d, n_traj * T)).astype(np.float32) for _ in range(5)]
    cu = [torch.from_numpy(x).cuda() for x in g]
    dt = 0.25
    Kx = K + 6 * ends
    Bm = rows(wbe, Kx, T, dt)
    tot = [g[0].astype(np.float64), g[1].astype(np.float64) + g[3], g[2].astype(np.float64) + g[4]]
    ref = sum(np.einsum("dns,sk->ndk", x.reshape(d, n_traj, T), b) for x, b in zip(tot, Bm))
    mag = sum(np.einsum("dns,sk->ndk", np.abs(x).reshape(d, n_traj, T), np.abs(b))
              for x, b in zip(tot, Bm))
    if ends:
        ref = np.concatenate([ref[..., 3:K + 2], ref[..., K + 2:].sum(-1, keepdims=True)], -1)
        mag = np.concatenate([mag[..., 3:K + 2], mag[..., K + 2:].sum(-1, keepdims=True)], -1)
        got, _ = wbe.bspline_backward_bc(cu[0], cu[1], cu[2], n_traj, K, T, dt, has_start=True,
                                         end_static=True, gqd_add=cu[3], gqdd_add=cu[4])
    else:
        got = wbe.bspline_backward(cu[0], cu[1], cu[2], n_traj, K, T, dt, gqd_add=cu[3],
                                   gqdd_add=cu[4])
    terms = 4 * T / (Kx - 3) + 4
    # each sample's three products and the added gradients, then the sum
    assert (np.abs(got.cpu().numpy() - ref) <= (terms + 12) * 6e-8 * mag + 1e-30).all()
