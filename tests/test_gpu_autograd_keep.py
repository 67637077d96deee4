"""The autograd functions keep the gradient of their forward pass: it is the evaluation kernel's
gradient to the bit, a second backward pass gives it again, an input changed in between is
reported, and a call that records nothing returns the same cost."""
import numpy as np
import pytest

from paper_2510_07674_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _inputs(kind):
    from paper_2510_07674_gb300 import autograd as A
    from paper_2510_07674_gb300 import spasm as S
    wl = scenes.make_problem("tower4", seed=3, B=2, O=10, W=8, N=64, M=16, P=4, Q=4)
    pr = S.Problem(wl)
    gen = torch.Generator().manual_seed(2)
    if kind == "place":
        x = torch.empty(8, 33, device="cuda")
        S.spasm_place_sample(pr, 33, 0, x, torch.empty(33, device="cuda"))
        g = torch.empty_like(x)
        S.spasm_place_eval(pr, 33, x, 1, torch.empty(33, device="cuda"), g)
        return pr, (lambda v: A.place_cost(pr, v, True)), x, g, lambda w: w[None, :]
    q = torch.tensor(wl.robot.q_home, dtype=torch.float32).repeat(33, pr.C, 1)
    q = (q + 0.3 * torch.randn(q.shape, generator=gen)).cuda()
    lam, mu = torch.rand(33, pr.NR, generator=gen).cuda(), 1 + torch.rand(33, generator=gen).cuda()
    q8, g = torch.zeros(33, pr.C, 8, device="cuda"), torch.empty(33, pr.C, 8, device="cuda")
    q8[:, :, :7] = q
    S.spasm_traj_eval(pr, 33, q8, lam, mu, torch.empty(33, device="cuda"), g)
    return pr, (lambda v: A.traj_cost(pr, v, lam, mu)), q8 if kind == "traj8" else q, g[:, :, : 8 if kind == "traj8" else 7], \
        lambda w: w[:, None, None]


@pytest.mark.parametrize("kind", ["place", "traj7", "traj8"])
def test_kept_gradient(kind):
    pr, f, x, g, spread = _inputs(kind)
    try:
        w = torch.linspace(-1, 2, 33, device="cuda")
        v = x.clone().requires_grad_(True)
        c = f(v)
        (g1,) = torch.autograd.grad(c, v, w, retain_graph=True)
        (g2,) = torch.autograd.grad(c, v, w)
        assert torch.equal(g1, g2) and torch.equal(g1, g * spread(w))
        with torch.no_grad():
            assert torch.equal(f(v), c.detach()) and torch.equal(f(x), c.detach())
        if kind != "traj7":   # traj7 is copied into padded rows
            c = f(v)
            with torch.no_grad():
                v += 1
            with pytest.raises(RuntimeError):
                c.sum().backward()
    finally:
        pr.close()
