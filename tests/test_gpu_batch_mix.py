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
