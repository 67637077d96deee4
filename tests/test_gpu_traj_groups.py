"""Particle groups of the trajectory kernels: a launch hands its particles to resident groups
(one or two per CTA) that take the next one from a counter when they are done.  A particle's
outputs are the same bits whatever the launch around it: alone, in launches that just fill or
just overflow the resident groups, under either shape, repeated on the same problem, with a
gradient buffer that is not 16-byte aligned, and for the largest sizes.  (The arithmetic itself
is compared with the oracle in test_gpu_stage2.py.)"""
import numpy as np
import pytest

from paper_2510_07674_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# blocks, cuboids, spheres, waypoints: short ragged segments (C - 1 not a multiple of 4 or 32), the
# largest problem (one particle per CTA only), all mask words of a small one
SIZES = [(1, 4, 0, 3), (2, 33, 0, 7), (3, 12, 5, 9), (4, 20, 0, 32), (16, 255, 64, 32)]


def _problem(B, O, sph, W):
    from paper_2510_07674_gb300 import spasm as S
    wl = scenes.make_problem("tower10", seed=B, B=B, O=O, W=W, N=256, M=64, Q=16, n_obstacle_spheres=sph)
    return S, S.Problem(wl)


def _lifted(S, pr, n):
    B = pr.B
    rng = np.random.default_rng(B)
    place = np.zeros((4, B, 4), np.float32)
    place[:, :, :2] = np.array([0.5, -0.3]) + rng.uniform(-0.02, 0.02, (4, B, 2))
    place[:, :, 2] = 0.025 + 0.05 * np.arange(B)
    place[:, :, 3] = rng.uniform(-3, 3, (4, B))
    q = torch.empty(n, pr.C, 8, device="cuda")
    S.spasm_lift(pr, n, torch.from_numpy(place).cuda(), 4, 0, q)
    return q


def _run(S, pr, q, lam, mu, steps=3):
    """Evaluation with gradient, then a short descent: every output."""
    n = len(q)
    L, g = torch.empty(n, device="cuda"), torch.empty(n, pr.C, 8, device="cuda")
    groups, h = torch.empty(n, 6, device="cuda"), torch.empty(n, pr.NR, device="cuda")
    S.spasm_traj_eval(pr, n, q, lam, mu, L, g, groups, h)
    q2, l2, m2 = q.clone(), lam.clone(), mu.clone()
    met, sat = torch.empty(n, 8, device="cuda"), torch.empty(n, device="cuda", dtype=torch.int32)
    S.spasm_traj_descend(pr, n, q2, l2, m2, steps, 0, met, sat)
    return [t.cpu().numpy() for t in (L, g, groups, h, q2, l2, m2, met, sat)]


def _same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("size", SIZES)
def test_a_particle_gives_the_same_bits_in_any_launch(size):
    S, pr = _problem(*size)
    try:
        n = 700 if size[0] < 16 else 330   # more than the resident groups of either shape
        q = _lifted(S, pr, n)
        gen = torch.Generator().manual_seed(1)
        lam, mu = torch.rand(n, pr.NR, generator=gen).cuda(), 1 + torch.rand(n, generator=gen).cuda()
        ref = _run(S, pr, q, lam, mu)
        _same(ref, _run(S, pr, q, lam, mu))   # the work counters start at zero again
        assert np.abs(ref[1]).max() > 0 and np.isfinite(ref[0]).all()
        for m in (1, 2, 303, 304, 305, 609):   # 2 x 152 groups of 8 warps, 4 x 152 of 4
            if m <= n:
                _same([r[:m] for r in ref], _run(S, pr, q[:m].contiguous(), lam[:m].contiguous(), mu[:m].contiguous()))
        for ppc in (1, 2):
            try:
                S.spasm_set_kernel_config(pr, 0, ppc)
            except S.SpasmError as e:
                assert e.status == -1 and ppc == 2   # two particles of the problem do not fit
                continue
            _same(ref, _run(S, pr, q, lam, mu))
    finally:
        pr.close()


def test_gradient_into_an_unaligned_buffer():
    S, pr = _problem(3, 12, 5, 9)
    try:
        q = _lifted(S, pr, 5)
        out = []
        for off in (0, 1):
            flat = torch.full((5 * pr.C * 8 + 1,), 7.0, device="cuda")
            L = torch.empty(5, device="cuda")
            S.spasm_traj_eval(pr, 5, q, None, None, L, flat[off: off + 5 * pr.C * 8])
            out.append(flat[off: off + 5 * pr.C * 8].cpu().numpy())
        assert np.array_equal(out[0], out[1])
    finally:
        pr.close()
