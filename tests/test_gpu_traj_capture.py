"""Trajectory calls captured into CUDA graphs share no scratch of their handle: graphs replayed side by
side on two streams, with direct calls on a third, give the bits of the calls made one by one.  (The
sizes take the captured launch through four, two and one particles per CTA, and more particles than
groups that are resident.)"""
import numpy as np
import pytest

from paper_2510_07674_gb300 import scenes
from test_gpu_traj_groups import _lifted, _problem, _run, _same

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _point_to_point(n):
    from paper_2510_07674_gb300 import spasm as S
    pr = S.Problem(scenes.make_p2p("p2p", seed=5, O=30, W=20, Q=16))
    rng = np.random.default_rng(4)
    ends = np.asarray(scenes.make_robot(7).q_home) + rng.uniform(-0.9, 0.9, (n, 2, 7))
    path = ends[:, :1] + np.linspace(0, 1, pr.C)[None, :, None] * (ends[:, 1:] - ends[:, :1])
    q = torch.zeros(n, pr.C, 8, device="cuda")
    q[:, :, :7] = torch.from_numpy(path.astype(np.float32)).cuda()
    return S, pr, q


@pytest.mark.parametrize("size, n", [(None, 700), ((1, 4, 0, 12), 1300), ((3, 12, 5, 9), 700), ((3, 255, 64, 32), 2500),
                                     ((6, 20, 0, 32), 700), ((16, 255, 64, 32), 330)])
def test_captured_calls_replayed_side_by_side(size, n):
    cap, a, b = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(cap):
        if size is None:
            S, pr, q = _point_to_point(2 * n)
        else:
            S, pr = _problem(*size)
            q = _lifted(S, pr, 2 * n)
        try:
            gen = torch.Generator().manual_seed(2)
            lam, mu = torch.rand(2 * n, pr.NR, generator=gen).cuda(), 1 + torch.rand(2 * n, generator=gen).cuda()
            torch.cuda.synchronize()
            ref = _run(S, pr, q, lam, mu)
            graphs, outs = [], []
            for part in (slice(0, n), slice(n, 2 * n)):
                qq, ll, mm = q[part].contiguous(), lam[part].contiguous(), mu[part].contiguous()
                L, g = torch.empty(n, device="cuda"), torch.empty(n, pr.C, 8, device="cuda")
                gr, h = torch.empty(n, 6, device="cuda"), torch.empty(n, pr.NR, device="cuda")
                met, sat = torch.empty(n, 8, device="cuda"), torch.empty(n, device="cuda", dtype=torch.int32)
                q2, l2, m2 = qq.clone(), ll.clone(), mm.clone()
                torch.cuda.synchronize()
                graph = torch.cuda.CUDAGraph()
                graph.capture_begin()
                S.spasm_traj_eval(pr, n, qq, ll, mm, L, g, gr, h)
                S.spasm_traj_descend(pr, n, q2, l2, m2, 3, 0, met, sat)
                graph.capture_end()
                graphs.append(graph)
                outs.append((L, g, gr, h, q2, l2, m2, met, sat))
                outs[-1] += (qq, ll, mm)
            with torch.cuda.stream(a):
                graphs[0].replay()
            with torch.cuda.stream(b):
                graphs[1].replay()
            direct = _run(S, pr, q, lam, mu)   # on the handle's own stream meanwhile
            torch.cuda.synchronize()
            _same(ref, direct)
            for part, out in zip((slice(0, n), slice(n, 2 * n)), outs):
                _same([r[part] for r in ref], [t.cpu().numpy() for t in out[:9]])
            S.spasm_synchronize(pr)
        finally:
            pr.close()
