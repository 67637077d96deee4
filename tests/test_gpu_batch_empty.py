"""A batch in which some problems have no placement: their items have no particle to run, so the
groups of the batched trajectory kernel drain them without any work in between, and the other
problems' results are those of their own solves, bit for bit."""
import numpy as np
import pytest

from paper_2510_07674_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _workloads():
    def empty(seed, Q):   # no placement can meet eps = 1e-9: stage 1 stops at its step budget with none
        return scenes.make_problem("tower4", seed=seed, B=2, O=6, W=6, N=512, M=128, Q=Q, eps=1e-9, max_steps=100)

    def full(seed, B, Q):
        return scenes.make_problem("tower4", seed=seed, B=B, O=12, W=10, N=1024, M=256, Q=Q)

    return [full(3, 2, 700), empty(1, 2500), full(4, 3, 517), empty(2, 1300)]


@pytest.mark.parametrize("config", [None, {"per_fetch": 1, "order": 1, "particles_per_cta": 1},
                                    {"per_fetch": 1, "order": 1, "particles_per_cta": 2},
                                    {"per_fetch": 64, "order": 0, "particles_per_cta": 2}])
def test_problems_without_a_placement_are_drained(config):
    from paper_2510_07674_gb300 import spasm as S
    wls = _workloads()
    alone = []
    for wl in wls:
        pr = S.Problem(wl)
        S.spasm_optimize(pr)
        alone.append(S.spasm_result(pr, allow_empty=True))
        pr.close()
    assert [a["n_found"] > 0 for a in alone] == [True, False, True, False]
    stream = torch.cuda.Stream()
    prs = [S.Problem(wl) for wl in wls]
    try:
        S.spasm_optimize_batch(prs, stream=stream.cuda_stream, config=config)
        for pr, a in zip(prs, alone):
            S.spasm_synchronize(pr)
            b = S.spasm_result(pr, allow_empty=True)
            assert b["n_found"] == a["n_found"]
            if a["n_found"]:
                for key in ("placements", "traj", "cost", "success"):
                    assert np.array_equal(a[key], b[key]), key
    finally:
        for pr in prs:
            pr.close()
