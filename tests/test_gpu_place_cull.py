"""Placement cost and gradient where the cull of the blocks and cubes below can go wrong: stacks and packings
around the 32 spheres (four blocks, four cubes) of one pass and the 32 cubes of one ballot, with neighbours
touching, overlapping and just apart, against the FP64 oracle (1e-4: the cost's and the gradient's FP32 rounding)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2510_07674_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RTOL = 1e-4


def _check(wl, xp, quad, fixed_z):
    from paper_2510_07674_gb300 import spasm as S
    orc, pr = O.Oracle(wl), S.Problem(wl)
    n, B = len(xp), pr.B
    x = torch.from_numpy(xp.reshape(n, 4 * B).T.copy()).float().cuda().contiguous()
    cost, grad = torch.empty(n, device="cuda"), torch.empty_like(x)
    S.spasm_place_eval(pr, n, x, quad, cost, grad, None, None)
    torch.cuda.synchronize()
    xs = x.cpu().double().numpy().T.reshape(n, B, 4)
    gs = grad.cpu().double().numpy().T.reshape(n, B, 4)
    touching = 0
    for p in range(n):
        c, g, t = orc.place_cost(xs[p], quad=bool(quad))
        touching += t[2] > 0
        assert abs(cost[p].item() - c) <= RTOL * max(abs(c), 1e-2), (p, cost[p].item(), c)
        keep = np.ones_like(g, dtype=bool)
        if fixed_z is not None:   # the sign of the height term at |z - z*| = 0 is the rounding of z*
            keep[np.abs(xs[p][:, 2] - fixed_z) < 1e-6, 2] = False
        assert np.linalg.norm((gs[p] - g)[keep]) <= RTOL * max(np.linalg.norm(g[keep]), 1e-2), p
    assert touching > n // 2


@pytest.mark.parametrize("quad", [0, 1])
@pytest.mark.parametrize("B", [2, 4, 5, 8, 9, 16])
def test_stacks(B, quad):
    wl = scenes.make_problem("tower10", seed=B, B=B, O=40, W=3, N=64, M=16, Q=4, P=4, n_obstacle_spheres=3)
    rng = np.random.default_rng(B)
    n = 48
    xp = O.Oracle(wl).place_sample(n)
    xp[:, :, :2] = xp[:, :1, :2] + rng.normal(0, 0.01, (n, B, 2))
    # heights from all blocks in one place to a stack with gaps
    z = np.sort(xp[:, :, 2], axis=1)
    xp[:, :, 2] = z[:, :1] + (z - z[:, :1]) * rng.uniform(0, 1.5, (n, 1))
    _check(wl, xp, quad, None)


@pytest.mark.parametrize("quad", [0, 1])
@pytest.mark.parametrize("gx", [4, 8, 9, 16])
def test_packings(gx, quad):
    wl = scenes.make_packing("tetris8", seed=gx, gx=gx, gy=4, N=64, M=16, P=4)
    rng = np.random.default_rng(gx)
    planted = np.repeat(wl.packing.planted[None], 24, 0)
    planted[:, :, :2] += rng.normal(0, 0.004, planted[:, :, :2].shape)
    planted[:, :, 3] += rng.normal(0, 0.04, planted[:, :, 3].shape)
    _check(wl, np.concatenate([planted, O.Oracle(wl).place_sample(24)]), quad, wl.packing.z_star)
