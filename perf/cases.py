"""The work that users of this library have it do, as cases to time.

A case is a plain dict; ``prepare`` makes what a caller has in hand before the call (a problem
handle, particles on the GPU), ``run`` makes one pass through the public entry points of
``paper_2510_07674_gb300.spasm`` / ``.autograd`` and returns the outputs whole, ``work`` counts
the bytes and operations a pass cannot do without and ``exact`` evaluates the same outputs in
64 bits with plain torch.  Sizes are those of the named workloads in ``scenes.py`` (towers of
1, 4 and 10 blocks, the 8-block packing, point to point, the heterogeneous batch) and the
ranges between them.

Kinds of case:

* ``place_grad``    stage-1 cost and gradient through ``autograd.place_cost`` (forward and
                    backward), for programs that put the placement cost into their own loss;
* ``place_select``  the head of Alg. 1: sample N placements, keep the M best;
* ``place_descend`` Alg. 1's descent of M placements (tower goal);
* ``pack_descend``  the same for the packing goal;
* ``traj_grad``     stage-2 objective and gradient through ``autograd.traj_cost``;
* ``traj_descend``  the augmented-Lagrangian descent of Q lifted trajectories (tower goal);
* ``p2p_descend``   the same for a point-to-point problem;
* ``check``         the FP64 feasibility check of caller-given trajectories;
* ``solve``         a whole solve: both stages and the result on the host;
* ``batch``         several problems of different sizes solved together.

Trajectory inputs are lifted here (damped-least-squares IK in 64 bits at the grasp and place
poses of a jittered tower, interpolated through perturbed via points), so that they depend on
the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_07674_gb300 import autograd, scenes
from paper_2510_07674_gb300 import spasm as S

F64 = torch.float64


# ------------------------------------------------------------------------------ the cases
def listed():
    return [
        # one gradient of a small placement set: a caller's own optimiser, latency bound
        dict(name="place_grad_1block_64", kind="place_grad", B=1, O=4, n=64, quadratic=True),
        # Alg. 1's sampling and elite selection at the 10-block workload's size
        dict(name="place_select_10blocks", kind="place_select", B=10, O=64, N=16384, M=4096),
        # its descent: 25 linear and 5 quadratic steps of the 4096 elites
        dict(name="place_descend_10blocks", kind="place_descend", B=10, O=64, n=4096, k_lin=25, k_quad=5),
        # the 8-block packing's descent (100 linear, 20 quadratic steps), the bulk of its solve
        dict(name="pack_descend_8blocks", kind="pack_descend", gx=8, gy=4, n=4096, k_lin=100, k_quad=20),
        # one gradient of a few short trajectories: latency bound
        dict(name="traj_grad_1block_64", kind="traj_grad", B=1, O=4, W=16, n=64, multipliers=False),
        # objective and gradient of a full set of 10-block trajectories (every configuration culled)
        dict(name="traj_grad_10blocks_4096", kind="traj_grad", B=10, O=64, W=32, n=4096, multipliers=True),
        # the 4-block workload's descent
        dict(name="traj_descend_4blocks", kind="traj_descend", B=4, O=20, W=32, n=2048, k=50),
        # point to point in clutter: one segment, every start path in collision
        dict(name="p2p_descend_1024", kind="p2p_descend", O=48, W=32, n=1024, k=50),
        # FP64 check of the 32 solutions a 10-block solve returns
        dict(name="check_10blocks_32", kind="check", B=10, O=64, W=32, n=32),
        # the smallest whole solve (an interactive pick and place)
        dict(name="solve_1block", kind="solve", base="tower1", B=1, O=4, N=256, M=64, Q=256, W=16, P=8),
        # the headline solve: the 10-block tower in clutter
        dict(name="solve_10blocks", kind="solve", base="tower10", B=10, O=64, N=16384, M=4096, Q=4096, W=32, P=32),
        # throughput form: problems of 1-10 blocks and 8-64 cuboids together
        dict(name="batch_12_mixed", kind="batch", problems=12, q_lo=1024, q_hi=4096, W=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["place_grad", "place_select", "place_descend", "pack_descend", "traj_grad", "traj_grad",
                       "traj_descend", "traj_descend", "p2p_descend", "check", "solve", "solve", "batch"])
    B, O, W = rng.randint(1, 10), rng.randint(4, 64), rng.randint(8, 32)
    if kind == "place_grad":
        return dict(kind=kind, B=B, O=O, n=_log_int(rng, 32, 16384), quadratic=rng.random() < 0.5)
    if kind == "place_select":
        N = _log_int(rng, 256, 16384)
        return dict(kind=kind, B=B, O=O, N=N, M=max(1, N // rng.choice([2, 3, 4, 7])))
    if kind == "place_descend":
        return dict(kind=kind, B=B, O=O, n=_log_int(rng, 64, 4096), k_lin=rng.randint(20, 40), k_quad=rng.randint(0, 10))
    if kind == "pack_descend":
        gx = rng.choice([4, 5, 6, 7, 8])
        return dict(kind=kind, gx=gx, gy=4, n=_log_int(rng, 64, 4096), k_lin=rng.randint(25, 100),
                    k_quad=rng.randint(5, 20))
    if kind == "traj_grad":
        return dict(kind=kind, B=B, O=O, W=W, n=_log_int(rng, 32, 4096), multipliers=rng.random() < 0.5)
    if kind == "traj_descend":
        return dict(kind=kind, B=B, O=O, W=W, n=_log_int(rng, 64, 4096), k=rng.randint(30, 50))
    if kind == "p2p_descend":
        return dict(kind=kind, O=rng.randint(12, 48), W=rng.randint(8, 64), n=_log_int(rng, 64, 2048),
                    k=rng.randint(30, 50))
    if kind == "check":
        return dict(kind=kind, B=B, O=O, W=W, n=rng.randint(1, 64))
    if kind == "solve":
        N = _log_int(rng, 256, 16384)
        return dict(kind=kind, base="tower10" if B > 1 else "tower1", B=B, O=O, N=N, M=max(64, N // 4),
                    Q=_log_int(rng, 256, 4096), W=W, P=rng.choice([8, 16, 32]))
    return dict(kind=kind, problems=rng.randint(2, 10), q_lo=256, q_hi=_log_int(rng, 512, 4096), W=W)


# ------------------------------------------------------------------------------ inputs
def _tower(case, seed, **kw):
    return scenes.make_problem("tower10", seed=seed, B=case["B"], O=case["O"], N=256, M=64, P=32, Q=64, **kw)


def _gen(seed, salt):
    g = torch.Generator(device="cpu")
    g.manual_seed(1_000_003 * seed + salt)
    return g


def _uniform(shape, lo, hi, gen):
    return lo + (hi - lo) * torch.rand(shape, generator=gen, dtype=F64)


def _sampled_placements(wl, n, gen):
    """n placements uniform over the goal box, as Alg. 1 samples them: (n, B, 4)."""
    sc, B = wl.scene, len(wl.scene.half)
    lo, hi = torch.zeros(B, 4, dtype=F64), torch.zeros(B, 4, dtype=F64)
    for i in range(B):
        z = max(float(sc.box[2]), float(sc.z_table + sc.half[i, 2])) if wl.packing is None else float(sc.box[2])
        lo[i] = torch.tensor([sc.box[0], sc.box[1], z, -math.pi])
        hi[i] = torch.tensor([sc.box[3], sc.box[4], sc.box[5], math.pi])
    return lo + (hi - lo) * torch.rand((n, B, 4), generator=gen, dtype=F64)


def _near_towers(wl, n, gen):
    """n nearly stacked towers, as stage 1 returns them: within 2 mm and 1 mm of height."""
    sc, B = wl.scene, len(wl.scene.half)
    x = torch.zeros(n, B, 4, dtype=F64)
    mid = torch.tensor([(sc.box[0] + sc.box[3]) / 2, (sc.box[1] + sc.box[4]) / 2], dtype=F64)
    x[:, :, :2] = mid + _uniform((n, 1, 2), -0.06, 0.06, gen) + _uniform((n, B, 2), -0.002, 0.002, gen)
    rest = torch.tensor(_z_targets(wl), dtype=F64)
    x[:, :, 2] = rest + _uniform((n, B), -0.001, 0.001, gen)
    x[:, :, 3] = _uniform((n, B), -math.pi, math.pi, gen)
    return x


def _z_targets(wl):
    z, out = float(wl.scene.z_table), []
    for h in wl.scene.half:
        out.append(z + float(h[2]))
        z += 2.0 * float(h[2])
    return out


def _lifted(wl, n, W, gen):
    """n trajectories (n, C, 7) in 64 bits: IK at every grasp and place pose from a perturbed
    home configuration, then start -> via -> goal on every segment."""
    p2p = wl.p2p
    B, n_t = len(wl.scene.half), (1 if p2p else 2 * len(wl.scene.half))
    dev = torch.device("cuda")
    init = torch.tensor(wl.scene.init, dtype=F64)
    half = torch.tensor(wl.scene.half, dtype=F64)
    target = torch.empty(n, n_t, 4, dtype=F64)
    if p2p:
        target[:, 0] = init[0]
    else:
        towers = _near_towers(wl, 32, gen)
        target[:, 0::2] = init
        target[:, 1::2] = towers[torch.arange(n) % 32]
        top = half[:, 2] + float(wl.scene.grasp_off)
        target[:, 0::2, 2] += top
        target[:, 1::2, 2] += top
    target[:, :, 3] += 0.5 * math.pi * torch.randint(0, 4, (n, n_t), generator=gen)
    home = torch.tensor(wl.robot.q_home, dtype=F64)
    q = _ik(wl.robot, target.to(dev), (home + _uniform((n, n_t, 7), -0.3, 0.3, gen)).to(dev))
    via = (home + _uniform((n, n_t, 7), -0.3, 0.3, gen)).to(dev)
    via = _to_limits(wl.robot, via)
    Sg = W - 1
    out = torch.empty(n, n_t * Sg + 1, 7, dtype=F64, device=dev)
    out[:, 0] = home.to(dev)
    m = Sg // 2
    for s in range(n_t):
        a = out[:, s * Sg].clone()
        for j in range(1, Sg + 1):
            if j <= m:
                out[:, s * Sg + j] = a + (j / m) * (via[:, s] - a)
            else:
                out[:, s * Sg + j] = via[:, s] + ((j - m) / (Sg - m)) * (q[:, s] - via[:, s])
    return out


def _to_limits(robot, q):
    lim = torch.tensor(robot.qlim, dtype=F64, device=q.device)
    return torch.minimum(torch.maximum(q, lim[:, 0]), lim[:, 1])


def _ik(robot, target, q, iterations=25):
    """Damped least squares to the top-down tool pose (x, y, z, yaw)."""
    c, s, zero = torch.cos(target[..., 3]), torch.sin(target[..., 3]), torch.zeros_like(target[..., 3])
    Rt = torch.stack([c, s, zero, s, -c, zero, zero, zero, zero - 1.0], -1).reshape(*c.shape, 3, 3)
    eye = 1e-4 * torch.eye(6, dtype=F64, device=q.device)
    for _ in range(iterations):
        R, o, Re, pe = _fk(robot, q)
        e_rot = 0.5 * torch.linalg.cross(Re.transpose(-1, -2), Rt.transpose(-1, -2), dim=-1).sum(-2)
        e = torch.cat([target[..., :3] - pe, e_rot], -1)
        z = torch.stack([R[k][..., :, 2] for k in range(1, 8)], -2)
        d = pe.unsqueeze(-2) - torch.stack(o[1:], -2)
        J = torch.cat([torch.linalg.cross(z, d, dim=-1), z], -1).transpose(-1, -2)   # (..., 6, 7)
        y = torch.linalg.solve(J @ J.transpose(-1, -2) + eye, e.unsqueeze(-1))
        q = _to_limits(robot, q + (J.transpose(-1, -2) @ y).squeeze(-1))
    return q


def _pad8(q):
    out = torch.zeros(*q.shape[:-1], 8, dtype=torch.float32, device="cuda")
    out[..., :7] = q.to("cuda").float()
    return out


def _inputs(case, seed):
    """The workload and the float32 particles of a kernel-level case, from the seed alone."""
    kind, gen = case["kind"], _gen(seed, 17)
    if kind == "pack_descend":
        wl = scenes.make_packing("tetris8", seed=seed, gx=case["gx"], gy=case["gy"], N=256, M=64)
        x = _sampled_placements(wl, case["n"], gen)
        return wl, x.reshape(case["n"], -1).t().float().cuda().contiguous()
    if kind in ("place_grad", "place_descend"):
        wl = _tower(case, seed, W=8)
        n = case["n"]
        x = _sampled_placements(wl, n, gen)
        if kind == "place_grad":   # a set in the middle of its refinement: half of it nearly stacked
            x[: n // 2] = _near_towers(wl, n // 2, gen)
        return wl, x.reshape(n, -1).t().float().cuda().contiguous()
    if kind == "place_select":
        return _tower(case, seed, W=8), None
    if kind == "p2p_descend":
        wl = scenes.make_p2p("p2p", seed=seed, O=case["O"], W=case["W"], Q=64)
    else:
        wl = _tower(case, seed, W=case["W"])
    return wl, _pad8(_lifted(wl, case["n"], case["W"], gen))


def _multipliers(case, NR, seed):
    """Multipliers and penalties in the range a descent reaches."""
    if not case["multipliers"]:
        return None, None
    gen = _gen(seed, 29)
    return _uniform((case["n"], NR), 0.0, 2.0, gen).float().cuda(), _uniform((case["n"],), 1.0, 8.0, gen).float().cuda()


def _batch_sizes(case):
    """Blocks, cuboids and trajectory particles of each problem of a batch (the sizes belong to
    the case, the scenes to the seed)."""
    rng = np.random.default_rng(np.random.SeedSequence([0xCA5E, case["problems"], case["q_hi"]]))
    return [dict(B=int(rng.integers(1, 11)), O=int(rng.integers(8, 65)),
                 Q=int(rng.integers(case["q_lo"], case["q_hi"] + 1))) for _ in range(case["problems"])]


def _batch_workloads(case, seed):
    return [scenes.make_problem("tower10", seed=1000 * (seed % 1000) + i, N=4096, M=1024, W=case["W"], **sizes)
            for i, sizes in enumerate(_batch_sizes(case))]


def _whole(result, P):
    """A solve's result at its full size: rows beyond the solutions found are zero."""
    out = dict(result)
    for key in ("traj", "cost", "success"):
        a = result[key]
        out[key] = np.zeros((P, *a.shape[1:]), a.dtype)
        out[key][: len(a)] = a
    return out


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.kind, st.case = case["kind"], case
    if st.kind == "solve":
        st.seed = seed
        keys = ("B", "O", "N", "M", "Q", "W", "P")
        st.problem = S.Problem(scenes.make_problem(case["base"], seed=seed, **{k: case[k] for k in keys}))
        return st
    if st.kind == "batch":
        st.stream = torch.cuda.Stream()
        st.workloads = _batch_workloads(case, seed)
        st.problems = [S.Problem(wl, stream=st.stream.cuda_stream) for wl in st.workloads]
        return st
    wl, x = _inputs(case, seed)
    st.problem, st.x = S.Problem(wl), x
    dev = torch.device("cuda")
    if st.kind == "place_grad":
        st.x.requires_grad_(True)
    elif st.kind == "place_select":
        st.x = torch.empty(4 * case["B"], case["N"], device=dev)
        st.cost = torch.empty(case["N"], device=dev)
        st.idx = torch.empty(case["M"], device=dev, dtype=torch.int32)
    elif st.kind in ("place_descend", "pack_descend"):
        st.buf = torch.empty_like(st.x)
        st.cost = torch.empty(case["n"], device=dev)
        st.sat = torch.empty(case["n"], device=dev, dtype=torch.int32)
    elif st.kind == "traj_grad":
        st.x.requires_grad_(True)
        st.lam, st.mu = _multipliers(case, st.problem.NR, seed)
    elif st.kind in ("traj_descend", "p2p_descend"):
        n = case["n"]
        st.buf = torch.empty_like(st.x)
        st.lam, st.mu = torch.empty(n, st.problem.NR, device=dev), torch.empty(n, device=dev)
        st.metrics, st.sat = torch.empty(n, 8, device=dev), torch.empty(n, device=dev, dtype=torch.int32)
    else:
        st.metrics = torch.empty(case["n"], 6, device=dev, dtype=F64)
        st.ok = torch.empty(case["n"], device=dev, dtype=torch.int32)
    return st


def run(st):
    case, kind = st.case, st.kind
    if kind == "solve":
        S.spasm_set_seed(st.problem, st.seed)
        S.spasm_optimize(st.problem)
        return _whole(S.spasm_result(st.problem, allow_empty=True), case["P"])
    if kind == "batch":
        for p, wl in zip(st.problems, st.workloads):
            S.spasm_set_seed(p, wl.params.seed)
        S.spasm_optimize_batch(st.problems, stream=st.stream.cuda_stream)
        return [_whole(S.spasm_result(p, allow_empty=True), wl.params.P) for p, wl in zip(st.problems, st.workloads)]
    if kind == "place_grad":
        cost = autograd.place_cost(st.problem, st.x, case["quadratic"])
        (grad,) = torch.autograd.grad(cost.sum(), st.x)
        return cost.detach(), grad
    if kind == "place_select":
        S.spasm_place_sample(st.problem, case["N"], 0, st.x, st.cost)
        S.spasm_select_topk(st.problem, case["N"], st.cost, case["M"], st.idx)
        return st.x, st.cost, st.idx
    if kind in ("place_descend", "pack_descend"):
        st.buf.copy_(st.x)   # the descent works in place
        S.spasm_place_descend(st.problem, case["n"], st.buf, case["k_lin"], case["k_quad"], st.cost, st.sat)
        return st.buf, st.cost, st.sat
    if kind == "traj_grad":
        L = autograd.traj_cost(st.problem, st.x, st.lam, st.mu)
        (grad,) = torch.autograd.grad(L.sum(), st.x)
        return L.detach(), grad
    if kind in ("traj_descend", "p2p_descend"):
        st.buf.copy_(st.x)
        S.spasm_traj_descend(st.problem, case["n"], st.buf, st.lam, st.mu, case["k"], 1, st.metrics, st.sat)
        return st.buf, st.lam, st.mu, st.metrics, st.sat
    S.spasm_traj_check(st.problem, case["n"], st.x, st.metrics, st.ok)
    return st.metrics, st.ok


# ------------------------------------------------------------------------------ work
_FK = 900      # kinematics of one configuration (seven sines and cosines, seven 3 x 4 products)
_CENTRE = 18   # one sphere centre
_TEST = 40     # one sphere against one cuboid
_CFG = 120     # update, path, limits and assembly of one configuration
_SPHERES = scenes.N_ARM_SPHERES


def _place_work(n, B, evaluations):
    """Every block sphere placed and tested once (against what it rests on), the tower terms."""
    return n * evaluations * (8 * B * (_CENTRE + _TEST) + 60 * B)


def _traj_work(n, C, B, steps):
    """The first evaluation places every sphere once; later ones move every configuration and
    need the kinematics of the grasp and place configurations and the placed blocks' tests (a
    configuration that stays clear of everything is known to without being looked at again)."""
    first = C * (_FK + _SPHERES * _CENTRE + _CFG)
    return n * (first + steps * (C * _CFG + 2 * B * _FK + 8 * B * (_CENTRE + _TEST)))


def work(case):
    kind = case["kind"]
    if kind in ("place_grad", "place_descend", "pack_descend"):
        B = case["B"] if "B" in case else case["gx"] * case["gy"] // 4
        n = case["n"]
        ev = 1 if kind == "place_grad" else case["k_lin"] + case["k_quad"] + 1
        per = 4 if kind == "pack_descend" else 1   # cells per block
        return {"bytes": 4 * n * (8 * B + 2), "flops": _place_work(n, B * per, ev)}
    if kind == "place_select":
        N, B = case["N"], case["B"]
        return {"bytes": 4 * (N * (4 * B + 1) + case["M"]), "flops": _place_work(N, B, 1)}
    if kind == "solve":
        return _solve_work(case["B"], case["N"], case["M"], case["Q"], case["W"], case["P"])
    if kind == "batch":
        total = {"bytes": 0, "flops": 0}
        for sizes in _batch_sizes(case):
            w = _solve_work(sizes["B"], 4096, 1024, sizes["Q"], case["W"], 32)
            total = {k: total[k] + w[k] for k in total}
        return total
    B = case.get("B", 1)
    C = case["W"] if kind == "p2p_descend" else 2 * B * (case["W"] - 1) + 1
    n, NR = case["n"], 9 * B + 3
    if kind == "traj_grad":
        return {"bytes": 4 * n * (16 * C + 1 + (NR + 1 if case["multipliers"] else 0)), "flops": _traj_work(n, C, B, 0)}
    if kind == "check":
        return {"bytes": n * (32 * C + 52), "flops": n * C * (_FK + _SPHERES * _CENTRE)}
    return {"bytes": 4 * n * (16 * C + NR + 10), "flops": _traj_work(n, C, B, case["k"])}


def _solve_work(B, N, M, Q, W, P, steps1=30, steps2=50):
    C = 2 * B * (W - 1) + 1
    flops = _place_work(N, B, 1) + _place_work(M, B, steps1 + 1) + _traj_work(Q, C, B, steps2)
    flops += P * C * (_FK + _SPHERES * _CENTRE)
    # what a solve hands over: the placements and the solutions
    return {"bytes": 4 * P * (4 * B + 7 * C + 2), "flops": flops}


# ------------------------------------------------------------------------------ 64 bits
def _const(a, dev):
    return torch.as_tensor(np.asarray(a), dtype=F64, device=dev)


def _fk(robot, q):
    """Frames 0..7 (rotations, origins) and the tool frame of q (..., 7), modified DH rows."""
    dev = q.device
    eye = torch.eye(3, dtype=F64, device=dev).expand(*q.shape[:-1], 3, 3)
    R, o = [eye], [torch.zeros(*q.shape[:-1], 3, dtype=F64, device=dev)]
    for k in range(7):
        a, al, d, th = (float(v) for v in robot.dh[k])
        ca, sa = math.cos(al), math.sin(al)
        c, s = torch.cos(th + q[..., k]), torch.sin(th + q[..., k])
        zero = torch.zeros_like(c)
        T = torch.stack([c, -s, zero, ca * s, ca * c, zero - sa, sa * s, sa * c, zero + ca], -1)
        t = torch.tensor([a, -sa * d, ca * d], dtype=F64, device=dev)
        o.append(o[-1] + R[-1] @ t)
        R.append(R[-1] @ T.reshape(*c.shape, 3, 3))
    ee = _const(robot.ee, dev)
    return R, o, R[7] @ ee[:3, :3], o[7] + R[7] @ ee[:3, 3]


def _norm(v):
    n2 = (v * v).sum(-1)
    pos = n2 > 0
    return torch.where(pos, torch.sqrt(torch.where(pos, n2, torch.ones_like(n2))), torch.zeros_like(n2))


def _pen(p, h, r):
    """Penetration of a sphere of radius r at p (box frame) into the box of half extents h."""
    q = p.abs() - h
    sd = _norm(q.clamp_min(0.0)) + q.amax(-1).clamp_max(0.0) - r
    return (-sd).clamp_min(0.0)


def _pen_env(scene, c, r):
    """(..., S) spheres against every environment obstacle: (..., S, O)."""
    cub = _const(scene.cuboid, c.device).reshape(-1, 15)
    R = cub[:, 3:12].reshape(-1, 3, 3)
    p = torch.einsum("oij,...oi->...oj", R, c.unsqueeze(-2) - cub[:, :3])
    return _pen(p, cub[:, 12:15], r.unsqueeze(-1))


def _pen_blocks(pose, half, c, r):
    """(..., S) spheres against upright boxes at pose (..., B, 4): (..., S, B)."""
    d = c.unsqueeze(-2) - pose[..., None, :, :3]
    cy, sy = torch.cos(pose[..., None, :, 3]), torch.sin(pose[..., None, :, 3])
    p = torch.stack([cy * d[..., 0] + sy * d[..., 1], -sy * d[..., 0] + cy * d[..., 1], d[..., 2]], -1)
    return _pen(p, half, r.unsqueeze(-1))


_SIGNS = [[(1.0 if m & (1 << a) else -1.0) for a in range(3)] for m in range(8)]


def _block_spheres(pose, local, r):
    """Spheres at `local` (k, 3) of each posed block: centres (..., B, k, 3), radii."""
    cy, sy = torch.cos(pose[..., 3])[..., None], torch.sin(pose[..., 3])[..., None]
    x = pose[..., 0:1] + cy * local[..., 0] - sy * local[..., 1]
    y = pose[..., 1:2] + sy * local[..., 0] + cy * local[..., 1]
    z = pose[..., 2:3] + local[..., 2].expand_as(x)
    return torch.stack([x, y, z], -1), r.expand(x.shape)


def _tower_terms(wl, pose, quadratic):
    """Support distances D (..., B), height errors e (..., B), collision sum and the largest
    penetration of placements (..., B, 4)."""
    dev, B = pose.device, pose.shape[-2]
    half = _const(wl.scene.half, dev)
    e = pose[..., 2] - torch.tensor(_z_targets(wl), dtype=F64, device=dev)
    D = []
    for i in range(B - 1):
        v = pose[..., i + 1:, :2].mean(-2) - pose[..., i, :2]
        cy, sy = torch.cos(pose[..., i, 3]), torch.sin(pose[..., i, 3])
        u = torch.stack([cy * v[..., 0] + sy * v[..., 1], -sy * v[..., 0] + cy * v[..., 1]], -1)
        D.append(_norm((u.abs() - half[i, :2]).clamp_min(0.0)))
    D.append(torch.zeros_like(e[..., 0]))
    signs = torch.tensor(_SIGNS, dtype=F64, device=dev)
    c, r = _block_spheres(pose, 0.5 * half[:, None, :] * signs, 0.5 * half.amin(-1)[:, None])
    env = _pen_env(wl.scene, c, r)
    below = _pen_blocks(pose, half, c.flatten(-3, -2), r.flatten(-2, -1)).unflatten(-2, (B, 8))
    j = torch.arange(B, device=dev)
    below = below * (j[None, None, :] < j[:, None, None]).to(F64)
    f = (lambda p: p * p) if quadratic else (lambda p: p)
    coll = f(env).sum((-1, -2, -3)) + f(below).sum((-1, -2, -3))
    maxpen = torch.maximum(env.amax((-1, -2, -3)), below.amax((-1, -2, -3)))
    return torch.stack(D, -1), e, coll, maxpen


def _place_cost(wl, pose, quadratic):
    D, e, coll, _ = _tower_terms(wl, pose, quadratic)
    p = wl.params
    return p.w_stable * D.sum(-1) + p.w_height * (e * e).sum(-1) + p.w_coll * coll


def _place_cost_grad(wl, pose, quadratic, chunk=512):
    costs, grads = [], []
    for x in pose.split(chunk):
        x = x.detach().requires_grad_(True)
        c = _place_cost(wl, x, quadratic)
        (g,) = torch.autograd.grad(c.sum(), x)
        costs.append(c.detach())
        grads.append(g)
    return torch.cat(costs), torch.cat(grads)


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 (Salmon et al., SC'11) of counter arrays, as four uint32 arrays."""
    c = [np.broadcast_to(np.asarray(v, np.uint64), np.broadcast(c0, c1).shape).copy() for v in (c0, c1, c2, c3)]
    k0, k1, m = key & 0xFFFFFFFF, (key >> 32) & 0xFFFFFFFF, np.uint64(0xFFFFFFFF)
    for _ in range(10):
        a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & m, (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & m]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _exact_select(case, wl):
    N, B, sc = case["N"], case["B"], wl.scene
    u = _philox(np.arange(B)[None, :], np.arange(N)[:, None], 0, 0, int(wl.params.seed))
    u = [(v >> np.uint64(8)).astype(np.float64) / 16777216.0 for v in u]
    zlo = np.maximum(sc.box[2], sc.z_table + sc.half[:, 2])
    x = np.stack([sc.box[0] + u[0] * (sc.box[3] - sc.box[0]), sc.box[1] + u[1] * (sc.box[4] - sc.box[1]),
                  zlo + u[2] * (sc.box[5] - zlo), -math.pi + u[3] * 2 * math.pi], -1)
    pose = torch.from_numpy(x).cuda()
    with torch.no_grad():
        cost = torch.cat([_place_cost(wl, c, False) for c in pose.split(512)])
    return [pose.reshape(N, -1).t().contiguous(), cost, None]   # the order of near ties has no 64-bit value


def _roll_pitch(R):
    return torch.atan2(R[..., 2, 1], R[..., 2, 2]), torch.atan2(-R[..., 2, 0], torch.hypot(R[..., 2, 1], R[..., 2, 2]))


def _held(wl, b, Re, pe):
    """Frame of the block held top-down by the tool: Re (..., 3, 3), pe (..., 3), block index b."""
    off = _const(wl.scene.half, pe.device)[b, 2] + float(wl.scene.grasp_off)
    flip = torch.tensor([1.0, -1.0, -1.0], dtype=F64, device=pe.device)
    return Re * flip, pe + off[..., None] * Re[..., :, 2]


def _trajectory_terms(wl, q, W):
    """Residuals, collision terms and metrics of tower trajectories q (n, C, 7)."""
    dev, B, Sg = q.device, len(wl.scene.half), W - 1
    C = q.shape[1]
    rb, half = wl.robot, _const(wl.scene.half, q.device)
    R, o, Re, pe = _fk(rb, q)
    t_grasp = torch.arange(B, device=dev) * 2 * Sg + Sg
    t_place = t_grasp + Sg
    blocks = torch.arange(B, device=dev)
    Rg, pg = _held(wl, blocks, Re[:, t_grasp], pe[:, t_grasp])
    Rp, pp = _held(wl, blocks, Re[:, t_place], pe[:, t_place])
    g_roll, g_pitch = _roll_pitch(Rg)
    p_roll, p_pitch = _roll_pitch(Rp)
    init = _const(wl.scene.init, dev)
    grasp = torch.cat([pg - init[:, :3], g_roll[..., None], g_pitch[..., None]], -1)
    tilt = torch.stack([p_roll, p_pitch], -1)
    placed = torch.cat([pp, torch.atan2(Rp[..., 1, 0], Rp[..., 0, 0])[..., None]], -1)   # (n, B, 4)
    D, e, coll, pm = _tower_terms(wl, placed, False)

    t = torch.arange(1, C, device=dev)
    seg = (t - 1) // Sg
    b = seg // 2
    held = ((seg % 2) == 1) & (t - seg * Sg < Sg)
    link = torch.as_tensor(np.asarray(rb.sphere_link), device=dev)
    sph = _const(rb.sphere, dev)
    Rl, ol = torch.stack(R, 2)[:, 1:], torch.stack(o, 2)[:, 1:]
    c_arm = torch.einsum("ntsij,sj->ntsi", Rl[:, :, link], sph[:, :3]) + ol[:, :, link]
    Rh, ph = _held(wl, b, Re[:, 1:], pe[:, 1:])
    loc = 0.5 * half[b][:, None, :] * torch.tensor(_SIGNS, dtype=F64, device=dev)
    c_blk = torch.einsum("ntij,tsj->ntsi", Rh, loc) + ph[:, :, None]
    pose = torch.where((blocks[None, :] < b[:, None])[None, :, :, None], placed[:, None], init[None, None])
    context = (blocks[None, :] != b[:, None]).to(F64)[None, :, None, :]
    c = torch.cat([c_arm, c_blk], 2)
    r = torch.cat([sph[:, 3].expand(C - 1, -1), (0.5 * half.amin(-1))[b][:, None].expand(-1, 8)], 1)
    r = r[None].expand(c.shape[:-1])
    env = _pen_env(wl.scene, c, r)
    blk = _pen_blocks(pose, half, c, r) * context
    mask = torch.ones(C - 1, c.shape[2], dtype=F64, device=dev)
    mask[:, len(link):] = held.to(F64)[:, None]
    total = (env.sum(-1) + blk.sum(-1)) * mask
    big = torch.maximum(env.amax(-1), blk.amax(-1)) * mask
    return dict(grasp=grasp, tilt=tilt, D=D, e=e, coll=coll, place_pen=pm, arm=total[..., : len(link)].sum((-1, -2)),
                blk=total[..., len(link):].sum((-1, -2)), maxpen=big.amax((-1, -2)))


def _objective(wl, q, W, lam, mu):
    p = wl.params
    T = _trajectory_terms(wl, q, W)
    w = lambda v: math.sqrt(v)   # noqa: E731
    h = torch.cat([w(p.w_start) * T["grasp"].flatten(1), w(p.w_start) * T["tilt"].flatten(1),
                   w(p.w_height) * T["e"], w(p.w_stable) * T["D"], w(p.w_coll) * T["coll"][:, None],
                   w(p.w_arm) * T["arm"][:, None], w(p.w_block) * T["blk"][:, None]], 1)
    lim = _const(wl.robot.qlim, q.device)
    path = ((q[:, 1:] - q[:, :-1]) ** 2).sum((-1, -2))
    over, under = (q[:, 1:] - lim[:, 1]).clamp_min(0.0), (lim[:, 0] - q[:, 1:]).clamp_min(0.0)
    jl = (over * over + under * under).sum((-1, -2))
    return p.w_path * path + p.w_jl * jl + (lam * h).sum(-1) + 0.5 * mu * (h * h).sum(-1)


def _per_chunk(case, wl):
    """Particles whose dense pair tables fit a few GB."""
    C = 2 * case["B"] * (case["W"] - 1) + 1
    return max(1, int(3.0e7 / (C * (_SPHERES + 8) * (case["O"] + 1 + case["B"]))))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "batch") or kind.endswith("descend"):
        # contacts that switch at rounding level make the end point of tens of descent steps depend on
        # the rounding: a 64-bit descent ends a few percent away, particle by particle
        return None
    wl, x = _inputs(case, seed)
    if kind == "place_select":
        return _exact_select(case, wl)
    if kind == "place_grad":
        pose = x.t().reshape(case["n"], -1, 4).to(F64)
        cost, grad = _place_cost_grad(wl, pose, case["quadratic"])
        return [cost, grad.reshape(case["n"], -1).t().contiguous()]
    q64, n, chunk = x[..., :7].to(F64), case["n"], _per_chunk(case, wl)
    if kind == "check":
        rows = []
        with torch.no_grad():
            for q in q64.split(chunk):
                T = _trajectory_terms(wl, q, case["W"])
                rows.append(torch.stack([T["maxpen"], (T["grasp"] ** 2).sum(-1).amax(-1), (T["tilt"] ** 2).sum(-1).amax(-1),
                                         T["place_pen"], T["D"].amax(-1), T["e"].abs().amax(-1)], -1))
        return [torch.cat(rows), None]
    NR = 9 * case["B"] + 3
    lam, mu = _multipliers(case, NR, seed)
    lam = torch.zeros(n, NR, dtype=F64, device="cuda") if lam is None else lam.to(F64)
    mu = torch.full((n,), float(wl.params.mu0), dtype=F64, device="cuda") if mu is None else mu.to(F64)
    Ls, gs = [], []
    for q, l, m in zip(q64.split(chunk), lam.split(chunk), mu.split(chunk)):
        q = q.detach().requires_grad_(True)
        L = _objective(wl, q, case["W"], l, m)
        (g,) = torch.autograd.grad(L.sum(), q)
        Ls.append(L.detach())
        gs.append(torch.nn.functional.pad(g, (0, 1)))
    # q[0] is the fixed home configuration: its row of the gradient is zero by definition
    grad = torch.cat(gs)
    grad[:, 0] = 0.0
    return [torch.cat(Ls), grad]
