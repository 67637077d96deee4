"""What a request of the service counts for against its budget: the problem's own buffers, which grow
with its particles, and nothing of the size of the GPU (the trajectory launches' scratch, which the
requests in flight share)."""
import pytest

from paper_2510_07674_gb300 import scenes


def _figures(B, W, Q):
    """Bytes of the stage-1 and result buffers, and of a trajectory particle."""
    C, N, M, P = 2 * B * (W - 1) + 1, 512, 128, 8
    fixed = 4 * (4 * B + 1) * N + 4 * (4 * B + 5) * M + P * C * 36 + 16 * B * P
    return C, dict(N=N, M=M, P=P, Q=Q), fixed, 32 * C + 4 * (9 * B + 3) + 48


@pytest.mark.parametrize("B, W", [(1, 16), (4, 32), (10, 32), (16, 32)])
def test_a_small_request_takes_little_of_the_budget(B, W):
    from paper_2510_07674_gb300 import spasm as S
    for Q in (8, 64, 2048):
        _, prm, fixed, particle = _figures(B, W, Q)
        got = S.spasm_problem_bytes(scenes.make_problem("tower10", seed=0, B=B, O=64, W=W, **prm))
        least = fixed + Q * particle
        # the rest: tables of the obstacles, constants, accumulators, 512-byte granules
        assert least < got < least + (96 << 10), (Q, got, least)


@pytest.mark.gpu
@pytest.mark.parametrize("B, W, groups", [(10, 32, 608), (1, 16, 1216)])
def test_a_problem_holds_its_bytes_and_the_scratch(B, W, groups):
    torch = pytest.importorskip("torch")
    from paper_2510_07674_gb300 import spasm as S
    from test_zz_no_alloc import _device_memory
    C, prm, _, _ = _figures(B, W, 64)
    wl = scenes.make_problem("tower10", seed=0, B=B, O=64, W=W, **prm)
    S.Problem(wl).close()
    torch.cuda.synchronize()
    before = _device_memory()[0]
    pr = S.Problem(wl)
    try:
        held = _device_memory()[0] - before
        assert abs(held - (S.spasm_problem_bytes(wl) + groups * 64 * C)) <= 64 << 10, held
    finally:
        pr.close()
