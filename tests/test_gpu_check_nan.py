"""The FP64 check refuses a trajectory with a joint that is not a number: its spheres and its
limit comparisons are all false, so that nothing else would."""
import numpy as np
import pytest

from test_gpu_check64 import _gpu_check, _planted

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_a_joint_that_is_not_a_number_is_refused():
    from paper_2510_07674_gb300 import spasm as S
    cs, _ = _planted()
    C = len(cs.q)
    qs = [cs.q.copy()]
    for t, j, v in [(1, 2, np.nan), (C // 2, 0, np.nan), (C - 1, 6, np.nan), (slice(1, C), slice(0, 7), np.nan),
                    (3, 1, np.inf)]:   # waypoints, the last place, all
        q = cs.q.copy()
        q[t, j] = v
        qs.append(q)
    pr = S.Problem(cs.pr)
    try:
        _, _, ok = _gpu_check(pr, qs)
        assert ok.tolist() == [1, 0, 0, 0, 0, 0]
    finally:
        pr.close()
