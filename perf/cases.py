"""The work that programs have this library do, as cases whose time and results can be measured.

A case is one pass of a Levenberg-Marquardt (LM) iteration through the public binding: the
parameters go in (``ba_set_params``), the reduced camera system is built (``ba_build_normal``), solved by
PCG or MCG, and the update comes out (``ba_get_delta``); or one loss-and-gradient evaluation of the
pose-grouping network.  Scenes come from the seeded generators (``synthetic.py``); every camera,
landmark and measurement depends on the seed.  The handle (the pattern of S, the work lists) is what a
program keeps over its LM iterations, so ``prepare`` makes it.

Tolerances.  A float64 handle solves to 1e-6, the benchmark's tolerance.  A mixed-precision handle
solves to 1e-9: to 1e-6 its one float32 sweep stops at an iterate that any reordering of a float32 sum
moves by 3e-5, while a second sweep on the double-float residual settles the digits of a float32,
which is also how such a handle is used when the update matters.  Those updates are handed on as
float32.
"""
import math

import numpy as np
import torch

from paper_2110_04015_gb300 import binding
from paper_2110_04015_gb300 import synthetic as sy

MAX_ITERS = 1000


def listed():
    return [
        # The smallest problems: 16 cameras, 1,000 landmarks, in the default precision; latency.
        {"name": "tiny_fp64_pcg", "kind": "solve", "scene": "tiny", "cams": 16, "pts": 1000, "precision": "fp64",
         "solver": "pcg", "dirs": 1, "tau": 0.0, "lam": 1e-4, "tol": 1e-6, "landmarks": False},
        # The same size in mixed precision, odd counts, MCG with the binding's default N and tau.
        {"name": "tiny_mixed_mcg", "kind": "solve", "scene": "tiny", "cams": 13, "pts": 777, "precision": "mixed",
         "solver": "mcg", "dirs": 8, "tau": 3.0, "lam": 1e-4, "tol": 1e-9, "landmarks": True},
        # A small dense collection in float64 (the parity tests' size).
        {"name": "dense150_fp64_mcg", "kind": "solve", "scene": "dense", "cams": 150, "pts": 20000,
         "precision": "fp64", "solver": "mcg", "dirs": 8, "tau": 3.0, "lam": 1e-4, "tol": 1e-6, "landmarks": True},
        # An ordinary collection in float64: build-bound.
        {"name": "dense601_fp64_pcg", "kind": "solve", "scene": "dense", "cams": 601, "pts": 90001,
         "precision": "fp64", "solver": "pcg", "dirs": 1, "tau": 0.0, "lam": 1e-4, "tol": 1e-6, "landmarks": True},
        # A video sequence (banded S that stays in L2): an LM iteration with the landmark update.
        {"name": "seq1000_mixed_pcg", "kind": "solve", "scene": "sequential", "cams": 1000, "pts": 100000,
         "precision": "mixed", "solver": "pcg", "dirs": 1, "tau": 0.0, "lam": 1e-4, "tol": 1e-9, "landmarks": True},
        # The same sequence by MCG, where nearly every step takes the local directions.
        {"name": "seq1000_mixed_mcg", "kind": "solve", "scene": "sequential", "cams": 1000, "pts": 100000,
         "precision": "mixed", "solver": "mcg", "dirs": 16, "tau": 10.0, "lam": 1e-4, "tol": 1e-9,
         "landmarks": False},
        # A clustered dense collection of 1,000 cameras with the landmark update.
        {"name": "dense1000_mixed_pcg", "kind": "solve", "scene": "dense", "cams": 1000, "pts": 400000,
         "precision": "mixed", "solver": "pcg", "dirs": 1, "tau": 0.0, "lam": 1e-4, "tol": 1e-9, "landmarks": True},
        # The benchmark's workload (1,936 cameras, 5.2 million observations) by PCG and by MCG.
        {"name": "dense1936_mixed_pcg", "kind": "solve", "scene": "dense", "cams": 1936, "pts": 1300000,
         "precision": "mixed", "solver": "pcg", "dirs": 1, "tau": 0.0, "lam": 1e-4, "tol": 1e-9, "landmarks": False},
        {"name": "dense1936_mixed_mcg", "kind": "solve", "scene": "dense", "cams": 1936, "pts": 1300000,
         "precision": "mixed", "solver": "mcg", "dirs": 16, "tau": 10.0, "lam": 1e-4, "tol": 1e-9,
         "landmarks": False},
        # Many uneven problems in the same launches.
        {"name": "batch16_mixed_mcg", "kind": "batch", "problems": 16, "cams_lo": 50, "cams_hi": 400,
         "pts_per_cam": 100, "precision": "mixed", "solver": "mcg", "dirs": 16, "tau": 10.0, "lam": 1e-4,
         "tol": 1e-9, "landmarks": False},
        # One loss-and-gradient evaluation of the grouping network on a training scene.
        {"name": "gnn_grad_240", "kind": "gnn", "scene": "sequential", "cams": 240, "pts": 14400,
         "precision": "mixed", "lam": 1e-4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: every size spread over the logarithm of its range."""
    lam = rng.choice([1e-4, 1e-4, 1e-3, 1e-2])
    solver = rng.choice(["pcg", "mcg"])
    dirs, tau = rng.choice([(8, 3.0), (16, 10.0), (4, 10.0), (11, 6.0)]) if solver == "mcg" else (1, 0.0)
    kind = rng.choice(["tiny", "dense64", "dense", "dense", "sequential", "sequential", "batch", "gnn"])
    if kind == "gnn":
        n = _log_int(rng, 80, 1000)
        return {"kind": "gnn", "scene": "sequential", "cams": n, "pts": 60 * n + rng.randrange(60),
                "precision": "mixed", "lam": lam}
    if kind == "batch":
        hi = _log_int(rng, 60, 400)
        return {"kind": "batch", "problems": _log_int(rng, 2, 24), "cams_lo": 50, "cams_hi": hi,
                "pts_per_cam": _log_int(rng, 30, 100), "precision": "mixed", "solver": solver, "dirs": dirs,
                "tau": tau, "lam": lam, "tol": 1e-9, "landmarks": rng.random() < 0.5}
    case = {"kind": "solve", "scene": kind, "precision": "mixed", "solver": solver, "dirs": dirs, "tau": tau,
            "lam": lam, "tol": 1e-9, "landmarks": rng.random() < 0.5}
    if kind == "tiny":
        n = _log_int(rng, 6, 48)
        case.update(cams=n, pts=n * _log_int(rng, 30, 120) + rng.randrange(30))
        if rng.random() < 0.5:
            case.update(precision="fp64", tol=1e-6)
    elif kind == "dense64":
        n = _log_int(rng, 60, 600)
        case.update(scene="dense", precision="fp64", tol=1e-6, cams=n, pts=n * _log_int(rng, 60, 150) + rng.randrange(60))
    elif kind == "dense":
        n = _log_int(rng, 60, 1900)
        case.update(cams=n, pts=n * _log_int(rng, 60, 650) + rng.randrange(60))
    else:
        n = _log_int(rng, 60, 1000)
        case.update(cams=n, pts=n * _log_int(rng, 60, 100) + rng.randrange(60))
    return case


# ---- inputs ---------------------------------------------------------------------------------------


def _scenes(case, seed):
    if case["kind"] == "batch":
        out = []
        for b in range(case["problems"]):   # uneven sizes, the same for every seed
            n = case["cams_lo"] + int((case["cams_hi"] - case["cams_lo"]) * (0.618034 * (b + 1) % 1.0))
            out.append(sy.dense(seed * 1000 + b, n_cams=n, n_pts=case["pts_per_cam"] * n,
                                n_clusters=max(1, n // 30), track_extra_mean=6.0, track_cap=min(200, n // 2),
                                p_uniform=0.3))
        return out
    n, m = case["cams"], case["pts"]
    if case["scene"] == "tiny":
        return [sy.tiny(seed, n_cams=n, n_pts=m, track_min=min(3, n), track_max=min(6, n))]
    if case["scene"] == "sequential":
        return [sy.sequential(seed, n_cams=n, n_pts=m)]
    return [sy.dense(seed, n_cams=n, n_pts=m, n_clusters=max(2, n // 30))]


def _rotation(w):
    """Rotation matrices of the angle-axis vectors w and the coefficients B, C of their Jacobians."""
    th2 = (w * w).sum(1)
    th = th2.sqrt()
    A, B, C = torch.sin(th) / th, (1 - torch.cos(th)) / th2, (th - torch.sin(th)) / (th2 * th)
    K = _skew(w)
    K2 = K @ K
    eye = torch.eye(3, dtype=w.dtype, device=w.device)
    R = eye + A[:, None, None] * K + B[:, None, None] * K2
    Jr = eye - B[:, None, None] * K + C[:, None, None] * K2
    return R, Jr


def _skew(v):
    z = torch.zeros_like(v[:, 0])
    return torch.stack([z, -v[:, 2], v[:, 1], v[:, 2], z, -v[:, 0], -v[:, 1], v[:, 0], z], 1).view(-1, 3, 3)


def _project(cams, pts, oc, op):
    R, _ = _rotation(cams[:, :3])
    P = torch.einsum("nij,nj->ni", R[oc], pts[op]) + cams[oc, 3:6]
    p = -P[:, :2] / P[:, 2:]
    n2 = (p * p).sum(1)
    return (cams[oc, 6] * (1 + cams[oc, 7] * n2 + cams[oc, 8] * n2 * n2))[:, None] * p


def _inputs(case, seed):
    """Cameras, landmarks, observations (int32) and measurements on the GPU, and the camera offsets."""
    scenes = _scenes(case, seed)
    cam_off, parts, n_pts = [0], [], 0
    for sc in scenes:
        to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        oc, op = to(sc.obs_cam).long(), to(sc.obs_pt).long()
        xy = _project(to(sc.cams_true), to(sc.pts_true), oc, op) + to(sc.noise)
        parts.append((to(sc.cams0), to(sc.pts0), oc + cam_off[-1], op + n_pts, xy))
        cam_off.append(cam_off[-1] + sc.n_cams)
        n_pts += sc.n_pts
    cams, pts, oc, op, xy = (torch.cat(v).contiguous() for v in zip(*parts))
    return cams, pts, oc.int(), op.int(), xy, cam_off


def prepare(case, seed):
    cams, pts, oc, op, xy, cam_off = _inputs(case, seed)
    batch = {"cam_off": cam_off} if case["kind"] == "batch" else {}
    problem = binding.Problem(cams, pts, oc, op, xy, precision=case["precision"], **batch)
    state = {"case": case, "problem": problem, "cams": cams, "pts": pts}
    if case["kind"] == "gnn":
        problem.ba_build_normal(case["lam"])
        state["net"] = binding.GNN(_network(seed))
    else:
        state["dxp"] = torch.zeros((cams.shape[0], 9), dtype=torch.float64, device="cuda")
        state["dxl"] = torch.zeros((pts.shape[0], 3), dtype=torch.float64, device="cuda") if case["landmarks"] else None
    return state


def run(state):
    case, p = state["case"], state["problem"]
    if case["kind"] == "gnn":
        loss, scores, grad = state["net"].ba_gnn_loss(p, grad=True)
        return {"loss": np.float32(loss), "scores": scores, "grad": grad}
    p.ba_set_params(state["cams"], state["pts"])
    p.ba_build_normal(case["lam"])
    if case["solver"] == "pcg":
        p.ba_solve_pcg(case["tol"], MAX_ITERS)
    else:
        p.ba_solve_mcg(case["tol"], MAX_ITERS, case["dirs"], case["tau"])
    p.ba_get_delta(state["dxp"], state["dxl"])
    out = {"dxp": state["dxp"]}
    if case["landmarks"]:
        out["dxl"] = state["dxl"]
    if case["precision"] == "mixed":
        out = {k: v.float() for k, v in out.items()}
    return out


def work(case):
    """Bytes: parameters, observations and measurements in, the update out.  Operations: the Jacobians, the
    products that form S (81 x 3 multiply-adds per pair of a landmark's observations), and the products
    with S of 20 iterations, fewer than any of these solves takes."""
    if case["kind"] == "batch":
        n_c = case["problems"] * (case["cams_lo"] + case["cams_hi"]) // 2
        n_l, track, width = case["pts_per_cam"] * n_c, 8.0, (case["cams_lo"] + case["cams_hi"]) / 2
    else:
        n_c, n_l = case["cams"], case["pts"]
        track, width = {"tiny": (4.5, n_c), "sequential": (7.0, 45.0), "dense": (4.0, n_c)}[case["scene"]]
    n_o = n_l * track
    pairs = n_o * (track - 1) / 2 * (1.5 if track in (4.0, 8.0) else 1.0)
    blocks = n_c * min(width, n_c) * (1 - math.exp(-2 * pairs / (n_c * min(width, n_c))))
    if case["kind"] == "gnn":
        layers = 2 * (8 + 64 + 64) * 64 * n_c + blocks * (8 + 64 + 64)
        return {"bytes": blocks * 324 + n_c * (72 + 4) + 2 * 4 * 17537, "flops": 3 * 2 * layers + 2 * 81 * blocks}
    nbytes = n_c * 72 + n_l * 24 + n_o * 24 + n_c * 72 + (n_l * 24 if case["landmarks"] else 0)
    return {"bytes": nbytes, "flops": 160 * n_o + 2 * 243 * pairs + 20 * 2 * 81 * blocks}


# ---- 64-bit values in plain torch -------------------------------------------------------------------


def _network(seed):
    """Glorot-uniform weights and zero biases of the network's layout (8 -> 64 -> 64 -> 64 -> 1)."""
    rs = np.random.RandomState(seed % (1 << 32))
    out = []
    for fan_in in (8, 64, 64):
        b = math.sqrt(6.0 / (fan_in + 64))
        out += [rs.uniform(-b, b, fan_in * 64), rs.uniform(-b, b, fan_in * 64), np.zeros(64)]
    b = math.sqrt(6.0 / 65)
    return np.concatenate(out + [rs.uniform(-b, b, 64), np.zeros(1)]).astype(np.float32)


def _reduced(cams, pts, oc, op, xy, lam):
    """S (dense), b~, and what the landmark update needs (W, V^-1, b_l) of one problem."""
    n_c, n_l, dt, dev = cams.shape[0], pts.shape[0], torch.float64, cams.device
    order = torch.argsort(op, stable=True)
    oc, op, xy = oc[order], op[order], xy[order]
    R, Jr = _rotation(cams[:, :3])
    Y = torch.einsum("nij,nj->ni", R[oc], pts[op])
    P = Y + cams[oc, 3:6]
    iz = 1 / P[:, 2]
    p = -P[:, :2] * iz[:, None]
    f, k1, k2 = cams[oc, 6], cams[oc, 7], cams[oc, 8]
    n2 = (p * p).sum(1)
    rho, drho = 1 + k1 * n2 + k2 * n2 * n2, k1 + 2 * k2 * n2
    r = (f * rho)[:, None] * p - xy
    E = f[:, None, None] * (rho[:, None, None] * torch.eye(2, dtype=dt, device=dev)
                            + 2 * drho[:, None, None] * p[:, :, None] * p[:, None, :])
    dp = torch.zeros((oc.numel(), 2, 3), dtype=dt, device=dev)
    dp[:, 0, 0] = dp[:, 1, 1] = -iz
    dp[:, :, 2] = -p * iz[:, None]
    D = E @ dp
    Jp = torch.empty((oc.numel(), 2, 9), dtype=dt, device=dev)
    Jp[:, :, :3] = -D @ _skew(Y) @ (R @ Jr)[oc]
    Jp[:, :, 3:6] = D
    Jp[:, :, 6] = rho[:, None] * p
    Jp[:, :, 7] = (f * n2)[:, None] * p
    Jp[:, :, 8] = (f * n2 * n2)[:, None] * p
    Jl = D @ R[oc]
    del dp, D, E

    def damped(blocks):
        d = torch.diagonal(blocks, dim1=1, dim2=2)
        d += lam * d.clamp(1e-6, 1e32)
        return blocks

    def add(n, idx, v):
        return torch.zeros((n,) + v.shape[1:], dtype=dt, device=dev).index_add_(0, idx, v)

    U = damped(add(n_c, oc, Jp.transpose(1, 2) @ Jp))
    Vi = torch.linalg.inv(damped(add(n_l, op, Jl.transpose(1, 2) @ Jl)))
    bp, bl = add(n_c, oc, torch.einsum("nij,ni->nj", Jp, r)), add(n_l, op, torch.einsum("nij,ni->nj", Jl, r))
    W = Jp.transpose(1, 2) @ Jl
    T = W @ Vi[op]
    bt = bp - add(n_c, oc, torch.einsum("nij,nj->ni", T, bl[op]))
    S = torch.zeros((n_c * n_c, 9, 9), dtype=dt, device=dev)
    d = 0
    while d < oc.numel():
        a = torch.nonzero(op[: op.numel() - d] == op[d:]).flatten()
        if a.numel() == 0:
            break
        for q in torch.split(a, 1 << 20):
            block = T[q] @ W[q + d].transpose(1, 2)
            S.index_add_(0, oc[q] * n_c + oc[q + d], block, alpha=-1.0)
            if d:
                S.index_add_(0, oc[q + d] * n_c + oc[q], block.transpose(1, 2).contiguous(), alpha=-1.0)
        d += 1
    S.view(n_c, n_c, 9, 9)[range(n_c), range(n_c)] += U
    S = S.view(n_c, n_c, 9, 9).transpose(1, 2).reshape(9 * n_c, 9 * n_c)
    return S, bt, (oc, op, W, Vi, bl)


def exact(case, seed):
    cams, pts, oc, op, xy, cam_off = _inputs(case, seed)
    oc, op = oc.long(), op.long()
    if case["kind"] == "gnn":
        return _exact_network(case, seed, cams, pts, oc, op, xy)
    dxp, dxl, first = [], [], 0
    for c0, c1 in zip(cam_off, cam_off[1:]):
        m = (oc >= c0) & (oc < c1)
        last = pts.shape[0] if c1 == cam_off[-1] else int(op[m].max()) + 1
        S, bt, (o, l, W, Vi, bl) = _reduced(cams[c0:c1], pts[first:last], oc[m] - c0, op[m] - first, xy[m], case["lam"])
        s = torch.diagonal(S).rsqrt()
        S *= s[:, None]
        S *= s[None, :]
        x = s * torch.cholesky_solve((-s * bt.flatten())[:, None], torch.linalg.cholesky(S))[:, 0]
        del S
        x = x.view(-1, 9)
        dxp.append(x)
        g = bl.index_add(0, l, torch.einsum("nij,ni->nj", W, x[o]))
        dxl.append(-torch.einsum("nij,nj->ni", Vi, g))
        first = last
    out = {"dxp": torch.cat(dxp)}
    if case["landmarks"]:
        out["dxl"] = torch.cat(dxl)
    return out


def _exact_network(case, seed, cams, pts, oc, op, xy):
    n = cams.shape[0]
    S, _, _ = _reduced(cams, pts, oc, op, xy, case["lam"])
    s = torch.diagonal(S).rsqrt()
    C = (s[:, None] * S * s[None, :]).view(n, 9, n, 9).square().sum((1, 3)).sqrt()
    C.fill_diagonal_(0)
    d = C.sum(1)
    R, _ = _rotation(cams[:, :3])
    centre = -torch.einsum("nji,nj->ni", R, cams[:, 3:6])
    centre = centre - centre.mean(0)
    centre = centre / centre.square().mean(0).sqrt()
    ld = torch.log1p(d)
    ld = ld - ld.mean()
    ld = ld / ld.square().mean().sqrt()
    H = torch.cat([centre, R[:, 2], ld[:, None], torch.ones_like(ld)[:, None]], 1)
    theta = torch.from_numpy(_network(seed)).double().cuda().requires_grad_()
    A, o = C / d[:, None], 0
    for fan_in in (8, 64, 64):
        k = fan_in * 64
        Ws, Wn, b = theta[o:o + k].view(fan_in, 64), theta[o + k:o + 2 * k].view(fan_in, 64), theta[o + 2 * k:o + 2 * k + 64]
        H, o = torch.relu(H @ Ws + (A @ H) @ Wn + b), o + 2 * k + 64
    scores = H @ theta[o:o + 64] + theta[o + 64]
    u = scores - (d @ scores) / d.sum()
    loss = (u @ (d * u) - u @ (C @ u)) / (u @ (d * u))
    loss.backward()
    return {"loss": loss.detach(), "scores": scores.detach(), "grad": theta.grad}
