"""Launch shapes of the trajectory kernel that only large launches take, and the point-to-point ones:
four particles per CTA at 49 to 192 configurations (several rounds of particles), and one, two and many
more particles than groups without blocks.  A particle's outputs are the bits it gives alone."""
import numpy as np
import pytest

from paper_2510_07674_gb300 import scenes
from test_gpu_traj_groups import _lifted, _problem, _run, _same

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _state(pr, n):
    gen = torch.Generator().manual_seed(3)
    return torch.rand(n, pr.NR, generator=gen).cuda(), 1 + torch.rand(n, generator=gen).cuda()


@pytest.mark.parametrize("size, n", [((2, 20, 0, 14), 2500), ((3, 12, 5, 32), 2433)])
def test_four_particles_per_cta_on_longer_trajectories(size, n):
    S, pr = _problem(*size)
    try:
        assert 48 < pr.C <= 192
        q = _lifted(S, pr, n)
        lam, mu = _state(pr, n)
        ref = _run(S, pr, q, lam, mu)
        assert np.isfinite(ref[0]).all()
        for m in (1, 300, 700):   # one and two per CTA
            _same([r[:m] for r in ref], _run(S, pr, q[:m].contiguous(), lam[:m].contiguous(), mu[:m].contiguous()))
        S.spasm_set_kernel_config(pr, 0, 1)
        _same(ref, _run(S, pr, q, lam, mu))
    finally:
        pr.close()


@pytest.mark.parametrize("O, W", [(12, 5), (48, 33), (40, 64)])
def test_point_to_point_groups(O, W):
    from paper_2510_07674_gb300 import spasm as S
    pr = S.Problem(scenes.make_p2p("p2p", seed=5, O=O, W=W, Q=16))
    try:
        n = 700
        rng = np.random.default_rng(W)
        home = np.asarray(scenes.make_robot(7).q_home)
        path = home + np.linspace(0, 1, pr.C)[None, :, None] * rng.uniform(-0.9, 0.9, (n, 1, 7))
        q = torch.zeros(n, pr.C, 8, device="cuda")
        q[:, :, :7] = torch.from_numpy(path.astype(np.float32)).cuda()
        lam, mu = _state(pr, n)
        ref = _run(S, pr, q, lam, mu)
        assert np.isfinite(ref[0]).all() and np.abs(ref[1]).max() > 0
        for m in (1, 2, 303, 304, 305, 609):
            _same([r[:m] for r in ref], _run(S, pr, q[:m].contiguous(), lam[:m].contiguous(), mu[:m].contiguous()))
        for ppc in (1, 2):
            S.spasm_set_kernel_config(pr, 0, ppc)
            _same(ref, _run(S, pr, q, lam, mu))
    finally:
        pr.close()
