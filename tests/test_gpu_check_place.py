"""The FP64 check where a placed block's pose cannot be had in FP32: its place configuration has
joints too large for an FP32 angle (on a robot with joint offsets, where the sum of the two rounds), or
holds the block's x axis vertical, so that its yaw hangs on the last bits.  The blocks' later
configurations reach into it; the metrics are the oracle's (1e-9 relative, as for every check).
And robots whose joint offsets, blocks whose yaws, are of many turns."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2510_07674_gb300 import scenes
from test_gpu_check64 import _compare, _float_limits, _gpu_check

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

B, W, N_TRAJ = 3, 8, 24
# horizontal part of the x axis: FP32 gives no yaw at all; and on both sides of the least that it is trusted
# with (half diagonal / extent of the scene, here about 0.01)
LEVEL = {"vertical": lambda rng: 2e-6, "tilted": lambda rng: 10.0 ** rng.uniform(-3.0, -1.0)}


def _workload(offsets=0.0):
    wl = scenes.make_problem("tower4", seed=4, B=B, O=0, W=W, N=64, M=16, P=4, Q=4, ik_mode=0)
    wl.scene.cuboid = np.zeros((0, 15))   # nothing but the blocks
    wl.scene.half = np.array([[0.04, 0.015, 0.025]] * B)
    wl.robot.dh[:, 3] = offsets
    return wl


def _upright(orc, rng, level):
    """A configuration whose tool x axis is vertical up to `level`: Newton steps on its horizontal part."""
    angle = rng.uniform(-np.pi, np.pi)
    target = level * np.array([np.cos(angle), np.sin(angle)])

    def res(q):
        return orc.fk(q)[1][:2, 0] - target
    q = rng.uniform(-1.0, 1.0, 7) + np.array([0, 0, 0, -1.5, 0, 1.0, 0])
    for _ in range(60):
        r = res(q)
        J = np.stack([(res(q + 1e-6 * e) - r) / 1e-6 for e in np.eye(7)], 1)
        q = q - np.clip(np.linalg.pinv(J, rcond=1e-6) @ r, -0.3, 0.3)
    assert np.abs(res(q)).max() < 1e-9
    return q


def _trajectories(kind, wl, orc):
    rng = np.random.default_rng(8)
    S = W - 1
    C = 2 * B * S + 1
    q = np.repeat(wl.robot.q_home[None, None], N_TRAJ, 0).repeat(C, 1)
    q += rng.uniform(-0.3, 0.3, q.shape)
    for p in range(N_TRAJ):
        t = 2 * S                                              # block 0's place configuration
        if kind == "large":
            far = rng.uniform(-1.0, 1.0, 7) + 2 * np.pi * rng.integers(20000, 40000, 7)
            q[p, t] = far.astype(np.float32)
            near = np.mod(q[p, t] + np.pi, 2 * np.pi) - np.pi   # the same angles
        else:
            q[p, t] = near = _upright(orc, rng, LEVEL[kind](rng))
        spread = 0.08 if kind == "large" else 0.01
        q[p, t + 1:] = near + rng.uniform(-spread, spread, (C - t - 1, 7))
    return q


@pytest.mark.parametrize("kind", ["large", "vertical", "tilted"])
def test_placed_blocks_that_fp32_cannot_place(kind):
    from paper_2510_07674_gb300 import spasm as S
    wl = _workload(np.array([0.3, -0.7, 1.1, -0.2, 0.9, -1.3, 0.5]) if kind == "large" else 0.0)
    orc = O.Oracle(_float_limits(wl))
    q = _trajectories(kind, wl, orc)
    pr = S.Problem(wl)
    try:
        q32, m, ok = _gpu_check(pr, q)
        _compare(orc, q32, m, ok)
        assert (m[:, 0] > 1e-3).sum() >= 12   # the arm is in the placed block
    finally:
        pr.close()


@pytest.mark.parametrize("offset", [50.0, 10000.0])
def test_joint_offsets_and_yaws_that_round_in_fp32(offset):
    """Joint offsets and initial yaws of many turns: their FP32 rounding moves every sphere and every
    block at its initial pose by more than the arithmetic's own rounding does."""
    from paper_2510_07674_gb300 import spasm as S
    turns = 2 * np.pi * np.round(offset / (2 * np.pi))
    wl = _workload(turns + np.array([0.3, -0.7, 1.1, -0.2, 0.9, -1.3, 0.5]))
    wl.scene.init[:, 3] += turns
    orc = O.Oracle(_float_limits(wl))
    rng = np.random.default_rng(3)
    C = 2 * B * (W - 1) + 1
    q = rng.uniform(-1.0, 1.0, (N_TRAJ, 1, 7)) + rng.uniform(-0.2, 0.2, (N_TRAJ, C, 7))
    q[:, 2 * (W - 1) + 1:] = q[:, [2 * (W - 1)]] + rng.uniform(-0.08, 0.08, (N_TRAJ, C - 2 * (W - 1) - 1, 7))
    pr = S.Problem(wl)
    try:
        q32, m, ok = _gpu_check(pr, q)
        _compare(orc, q32, m, ok)
        assert (m[:, 0] > 1e-3).sum() >= 12
    finally:
        pr.close()
