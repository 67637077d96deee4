"""The FP64 check's FP32 screen: trajectories on which picking the configurations to repeat in
FP64 could go wrong give the oracle's metrics all the same (1e-9 relative, as for every check):
all configurations tied, obstacle spheres, nothing near, joints too large for an FP32 angle,
one configuration, the last of a ragged slice."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2510_07674_gb300 import scenes
from test_gpu_check64 import _compare, _float_limits, _gpu_check

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _case(kind):
    rng = np.random.default_rng(5)
    B, O_, sph, W = {"spheres": (3, 8, 20, 9), "clear": (1, 0, 0, 5), "last": (2, 10, 0, 18)}.get(kind, (2, 12, 0, 8))
    wl = scenes.make_problem("tower4", seed=4, B=B, O=O_, W=W, N=64, M=16, P=3, Q=4, n_obstacle_spheres=sph)
    lim = wl.robot.qlim
    C = 2 * B * (W - 1) + 1
    q = np.repeat(wl.robot.q_home[None, None], 7, 0).repeat(C, 1)
    if kind == "clear":
        wl.scene.cuboid = np.zeros((0, 15))
    elif kind == "tied":
        q += rng.uniform(-0.6, 0.6, (7, 1, 7))             # every configuration the same
    elif kind == "large":
        q += rng.uniform(-0.4, 0.4, q.shape)
        q[:, ::5, 0] += 6 * np.pi                          # outside the limits and beyond the FP32 range
    elif kind == "last":
        q[:, -1] += rng.uniform(-0.9, 0.9, (7, 7))         # only the last configuration moves
    else:
        q += rng.uniform(-0.8, 0.8, q.shape)
    if kind != "large":
        q = np.clip(q, lim[:, 0] + 1e-3, lim[:, 1] - 1e-3)
    return wl, q


@pytest.mark.parametrize("kind", ["tied", "spheres", "clear", "large", "last", "random"])
def test_screened_check_matches_oracle(kind):
    from paper_2510_07674_gb300 import spasm as S
    wl, q = _case(kind)
    pr = S.Problem(wl)
    try:
        orc = O.Oracle(_float_limits(wl))
        for _ in range(2):   # the accumulators are clear again for the second call
            q32, m, ok = _gpu_check(pr, q)
            _compare(orc, q32, m, ok)
        if kind == "clear":
            assert np.all(m[:, 0] == 0.0)
        elif kind != "last":
            assert m[:, 0].max() > 1e-3   # something is penetrated
    finally:
        pr.close()
