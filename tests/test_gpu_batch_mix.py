"""Batches whose groups change problems often: each change restages another problem's constants,
tables and boxes over those of the last one, in memory laid out by other sizes.  Every problem's result
is that of its own solve, bit for bit."""
import numpy as np
import pytest

from paper_2510_07674_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _alone(wls):
    from paper_2510_07674_gb300 import spasm as S
    out = []
    for wl in wls:
        pr = S.Problem(wl)
        S.spasm_optimize(pr)
        out.append(S.spasm_result(pr, allow_empty=True))
        pr.close()
    assert any(r["n_found"] for r in out)
    return out


def _same(a, b):
    assert a["n_found"] == b["n_found"]
    for key in ("traj", "cost", "success") + (("placements",) if a["n_found"] else ()):
        assert np.array_equal(a[key], b[key]), key


def _batch(wls, alone, config, times=1):
    from paper_2510_07674_gb300 import spasm as S
    stream = torch.cuda.Stream()
    for _ in range(times):
        prs = [S.Problem(wl) for wl in wls]
        try:
            S.spasm_optimize_batch(prs, stream=stream.cuda_stream, config=config)
            for pr, a in zip(prs, alone):
                S.spasm_synchronize(pr)
                _same(a, S.spasm_result(pr, allow_empty=True))
        finally:
            for pr in prs:
                pr.close()


@pytest.mark.parametrize("ppc", [1, 2])
def test_groups_that_restage_other_problems(ppc):
    """Four problems a group: tables of 1 to 256 cuboids and 0 to 64 spheres, 1 to 4 blocks."""
    sizes = [(1, 255, 0), (4, 3, 64), (2, 0, 1), (3, 97, 12), (1, 5, 0), (4, 64, 33), (2, 200, 7), (3, 1, 0)]
    wls = [scenes.make_problem("tower4", seed=60 + i, B=B, O=O, W=6, N=512, M=128, Q=304, n_obstacle_spheres=sph)
           for i, (B, O, sph) in enumerate(sizes)]
    _batch(wls, _alone(wls), {"per_fetch": 1, "order": 1, "particles_per_cta": ppc})


def _two_shapes():
    """Problems on both sides of the rule that leaves a batch its launch shapes (6 blocks), so that two
    launches run side by side, with one that has no placement."""
    def wl(i, B, Q, **kw):
        return scenes.make_problem("tower10", seed=80 + i, B=B, O=16, W=8, N=2048, M=512, Q=Q, P=8, **kw)

    return [wl(0, 2, 517), wl(1, 8, 300), wl(2, 4, 700), wl(3, 10, 333), wl(4, 2, 900, eps=1e-9, max_steps=100),
            wl(5, 7, 130), wl(6, 6, 256)]


def test_two_launch_shapes_side_by_side():
    wls = _two_shapes()
    alone = _alone(wls)
    assert sum(r["n_found"] > 0 for r in alone) >= 4
    _batch(wls, alone, None, times=2)


def test_service_with_two_launch_shapes_in_flight():
    from paper_2510_07674_gb300 import spasm as S
    wls = _two_shapes()
    alone = _alone(wls)
    sv = S.Server(budget_bytes=4 << 30, max_inflight=len(wls))
    try:
        tickets = [S.spasm_server_submit(sv, wl) for wl in wls + wls]   # the second half joins later epochs
        for t in tickets:
            S.spasm_server_wait(sv, t, 300.0)
        got = [S.spasm_server_result(sv, t) for t in tickets]
        st = S.spasm_server_get_stats(sv)
    finally:
        sv.close()
    for a, b in zip(alone + alone, got):
        assert b["status"] == (0 if a["n_found"] else -4)
        _same(a, b)
    assert st["requests_in_epochs"] > st["epochs"], st
