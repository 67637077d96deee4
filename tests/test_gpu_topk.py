"""spasm_select_topk where its gathering and its sort can go wrong: sizes around the 32, 64 and 1024 keys that
a warp, a warp's sort and a block take at a time, and keys of which many, all or none equal the k-th smallest."""
import numpy as np
import pytest

from paper_2510_07674_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 31, 33, 64, 256, 1023, 1025, 4097, 16384])
@pytest.mark.parametrize("kind", ["distinct", "ties", "equal", "nan", "special"])
def test_topk_is_the_stable_argsort(n, kind):
    from paper_2510_07674_gb300 import spasm as S

    rng = np.random.default_rng(n)
    c = {"distinct": rng.permutation(n) - 0.5 * n,
         "ties": rng.integers(0, 3, n) * 1.0,
         "equal": np.zeros(n),
         "nan": np.where(rng.random(n) < 0.7, np.nan, rng.random(n)),
         "special": rng.choice([np.inf, -np.inf, np.nan, -0.0, 0.0, 3e38, -1e-42], n)}[kind].astype(np.float32)
    ref = np.argsort(c, kind="stable")     # NaN last, -0 and 0 equal, ties by index
    pr = S.Problem(scenes.make_problem("tower1", seed=0))
    cost = torch.from_numpy(c).cuda()
    for k in sorted({1, min(n, 32), min(n, 65), (n + 1) // 2, min(n, 8192)}):
        idx = torch.full((k,), -1, dtype=torch.int32, device="cuda")
        S.spasm_select_topk(pr, n, cost, k, idx)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(idx.cpu().numpy(), ref[:k])
