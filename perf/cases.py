"""Timed cases of the STBA solver: what its users run, through the public entry points, over the range of sizes.

A case is one problem (a seeded synthetic scene: cameras, points, pixel observations) and what a program does
with it: `iterate` runs LM iterations of a kept context from given parameters and takes the parameters back;
`adjoint` records them and differentiates the result; `cost` evaluates F(x) on caller-owned device arrays.
Scenes have the shapes of the repository's configurations: a ring of cameras around an object, a photo
collection on a hemisphere with Zipf track lengths, and a vehicle's trajectory with tracks of consecutive
frames.  Mixed-precision cases hand the parameters (or gradients) back as FP32 tensors, as the differentiable
entry point does for FP32 inputs; FP64 cases hand back FP64.
"""
import math

import numpy as np
import torch

from paper_2008_00446_gb300 import stba

HALF_W, HALF_H = 320.0, 240.0   # 640 x 480 images


def _case(name, scene, cams, points, lmax=50, cap=100, clusters="joins", precision="mixed", entry="iterate", iters=5,
          lambda0=0.05, huber=0.0, solver="clusters"):
    c = dict(scene=scene, cams=cams, points=points, lmax=lmax, cap=cap, clusters=clusters, precision=precision,
             entry=entry, iters=iters, lambda0=lambda0, huber=huber, solver=solver)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a local window of a tracker, refined in a few iterations
        _case("window_10", "ring", 10, 200, cap=5, clusters="spatial", iters=3, lambda0=0.3),
        # the 30-camera ring in FP64, the library's default precision, with fixed clusters
        _case("ring_30_fp64", "ring", 30, 2000, cap=10, clusters="spatial", precision="fp64", iters=5),
        # FP64 at clusters of full size, with the heavy damping that turns the steepest-descent correction on
        _case("photos_300_fp64", "hemisphere", 300, 30_000, clusters="joins", precision="fp64", iters=2, lambda0=0.5),
        # the benchmark's workload: a photo collection, a new clustering before every iteration (Algorithm 1)
        _case("photos_1000_draws", "hemisphere", 1000, 200_000, iters=5),
        # the same with a fixed spatial partition and the Huber loss of the paper's experiments
        _case("photos_1000_huber", "hemisphere", 1000, 200_000, clusters="spatial", iters=5, huber=0.5),
        # sequential frames: uneven contiguous clusters of 20 to 300 cameras, re-used every iteration
        _case("drive_2000_uneven", "drive", 2000, 200_000, lmax=20, cap=300, clusters="uneven", iters=3, lambda0=0.09),
        # all cameras in one dense system: plain LM with the full reduced camera system
        _case("photos_400_dense", "hemisphere", 400, 40_000, cap=400, clusters="spatial", iters=2),
        # a large collection: more clusters than the GPU factors at once
        _case("photos_6000_draws", "hemisphere", 6000, 900_000, lmax=80, iters=2),
        # differentiable use: a recorded solve and its reverse pass
        _case("adjoint_500", "hemisphere", 500, 50_000, clusters="spatial", entry="adjoint", iters=4, lambda0=0.3),
        # the conjugate-gradient solvers: the full system, and the clustered one
        _case("photos_1000_pcg", "hemisphere", 1000, 200_000, iters=1, lambda0=1e-2, clusters="spatial",
              solver="pcg_full"),
        _case("photos_500_pcg_split", "hemisphere", 500, 50_000, iters=1, lambda0=1e-2, clusters="spatial",
              solver="pcg_clusters"),
        # F(x) alone, without allocation, on arrays the caller holds
        _case("cost_1000", "hemisphere", 1000, 200_000, precision="fp64", entry="cost"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["window", "ring64", "photos64", "photos", "photos", "photos", "huber", "drive", "drive", "dense",
                       "adjoint", "pcg", "split", "cost"])
    if kind == "window":
        m = _log(rng, 10, 40)
        return _case("", "ring", m, _log(rng, 20 * m, 100 * m), cap=max(3, m // rng.randint(1, 4)), clusters="spatial",
                     iters=rng.randint(1, 3), lambda0=0.3)
    if kind == "ring64":
        m = _log(rng, 10, 60)
        return _case("", "ring", m, _log(rng, 25 * m, 100 * m), cap=rng.randint(5, 20), clusters="spatial",
                     precision="fp64", iters=rng.randint(1, 5))
    m = _log(rng, 150, 3000)
    n = _log(rng, 100 * m, 220 * m)
    cap = rng.choice([40, 70, 100, 100, 150])
    lam = rng.choice([0.05, 0.09, 0.2])
    if kind == "photos64":
        m = _log(rng, 100, 400)
        return _case("", "hemisphere", m, _log(rng, 60 * m, 150 * m), cap=rng.choice([40, 70, 100]), precision="fp64",
                     iters=2, lambda0=lam)
    if kind == "photos":
        return _case("", "hemisphere", m, n, lmax=rng.randint(20, 80), cap=cap, clusters=rng.choice(["joins", "spatial"]),
                     iters=rng.randint(1, 4), lambda0=lam)
    if kind == "huber":
        return _case("", "hemisphere", m, n, lmax=rng.randint(20, 80), cap=cap, clusters="spatial",
                     iters=rng.randint(1, 4), huber=rng.choice([0.5, 1.0, 2.0]))
    if kind == "drive":
        m = _log(rng, 200, 2000)
        return _case("", "drive", m, _log(rng, 50 * m, 100 * m), lmax=rng.randint(8, 20), cap=rng.randint(100, 300),
                     clusters="uneven", iters=rng.randint(1, 3), lambda0=lam)
    if kind == "dense":
        m = _log(rng, 60, 400)
        return _case("", "hemisphere", m, _log(rng, 60 * m, 120 * m), cap=m, clusters="spatial", iters=rng.randint(1, 2))
    if kind == "adjoint":
        m = _log(rng, 100, 600)
        return _case("", "hemisphere", m, _log(rng, 60 * m, 120 * m), cap=rng.choice([40, 70, 100]), clusters="spatial",
                     entry="adjoint", iters=rng.randint(2, 4), lambda0=rng.choice([0.2, 0.3, 1.0]))
    if kind in ("pcg", "split"):
        m = _log(rng, 150, 1000)
        return _case("", "hemisphere", m, _log(rng, 100 * m, 200 * m), cap=cap, clusters="spatial", iters=1, lambda0=1e-2,
                     solver="pcg_full" if kind == "pcg" else "pcg_clusters")
    return _case("", "hemisphere", m, n, lmax=rng.randint(20, 80), precision="fp64", entry="cost")


# ------------------------------------------------------------------------------------------------------
# scenes, made on the GPU from the seed
def _look(fwd):
    """World-to-camera rotations with the viewing directions fwd (k, 3), +z up, as angle-axis vectors."""
    up = torch.zeros_like(fwd)
    up[:, 2] = 1.0
    up[fwd[:, 2].abs() > 0.999] = torch.tensor([0.0, 1.0, 0.0], dtype=fwd.dtype, device=fwd.device)
    right = torch.linalg.cross(fwd, up)
    right = right / right.norm(dim=1, keepdim=True)
    R = torch.stack([right, torch.linalg.cross(fwd, right), fwd], dim=1)
    # quaternion from the largest of its four components, then angle and axis
    t = R.diagonal(dim1=1, dim2=2)
    q2 = torch.stack([1 + t.sum(1), 1 + 2 * t[:, 0] - t.sum(1), 1 + 2 * t[:, 1] - t.sum(1), 1 + 2 * t[:, 2] - t.sum(1)], 1)
    a, b, c = R[:, 2, 1], R[:, 0, 2], R[:, 1, 0]
    d, e, f = R[:, 1, 2], R[:, 2, 0], R[:, 0, 1]
    rows = torch.stack([torch.stack([q2[:, 0], a - d, b - e, c - f], 1), torch.stack([a - d, q2[:, 1], c + f, b + e], 1),
                        torch.stack([b - e, c + f, q2[:, 2], a + d], 1), torch.stack([c - f, b + e, a + d, q2[:, 3]], 1)], 1)
    q = rows[torch.arange(len(R), device=R.device), q2.argmax(1)]
    q = q / q.norm(dim=1, keepdim=True)
    q = torch.where(q[:, :1] < 0, -q, q)
    s = q[:, 1:].norm(dim=1, keepdim=True)
    return 2 * torch.atan2(s, q[:, :1]) * q[:, 1:] / s


def _rotate(w, X):
    th = w.norm(dim=-1, keepdim=True)
    k = w / th
    return (X * th.cos() + torch.linalg.cross(k.expand_as(X), X) * th.sin() +
            k * (k * X).sum(-1, keepdim=True) * (1 - th.cos()))


def _pixels(c, X):
    Y = _rotate(c[..., :3], X) + c[..., 3:6]
    x = Y[..., :2] / torch.where(Y[..., 2:] > 1e-9, Y[..., 2:], torch.ones_like(Y[..., 2:]))
    r2 = (x * x).sum(-1, keepdim=True)
    uv = c[..., 6:7] * (1 + r2 * (c[..., 7:8] + r2 * c[..., 8:9])) * x
    return uv, Y[..., 2]


def _inside(uv, z, zmin):
    return (z > zmin) & (uv[..., 0].abs() < HALF_W) & (uv[..., 1].abs() < HALF_H)


def _problem(case, seed):
    """cameras, points (initial), obs_cam, obs_pt, obs_uv as CUDA tensors; the camera centres; a NumPy generator."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(1_000_003 * (int(seed) + 1) + case["cams"])
    m, n, lmax = case["cams"], case["points"], case["lmax"]

    def rand(*shape):
        return torch.rand(shape, generator=g, device=dev, dtype=torch.float64)

    def randn(*shape):
        return torch.randn(shape, generator=g, device=dev, dtype=torch.float64)

    kind = case["scene"]
    phi = 2 * math.pi * torch.arange(m, device=dev, dtype=torch.float64) / m
    if kind == "ring":
        C = torch.stack([10 * phi.cos(), 10 * phi.sin(), 0 * phi], 1)
        fwd = -C / 10
    elif kind == "hemisphere":
        radius = 20.0 * math.sqrt(max(1.0, m / 2000.0))   # larger collections cover a larger site
        cz, az = rand(m), 2 * math.pi * rand(m)
        sz = (1 - cz * cz).sqrt()
        C = radius * torch.stack([sz * az.cos(), sz * az.sin(), cz], 1)
        fwd = -C / radius
    else:   # a closed path with three self-crossings, 0.4 m between frames
        P = torch.stack([phi.sin() + 2 * (2 * phi).sin(), phi.cos() - 2 * (2 * phi).cos()], 1)
        D = torch.stack([phi.cos() + 4 * (2 * phi).cos(), -phi.sin() + 4 * (2 * phi).sin()], 1)
        C = torch.cat([P * (0.4 * m / 23.0), torch.full((m, 1), 1.5, device=dev, dtype=torch.float64)], 1)
        fwd = torch.cat([D / D.norm(dim=1, keepdim=True), torch.zeros((m, 1), device=dev, dtype=torch.float64)], 1)
    w = _look(fwd)
    true = torch.cat([w, -_rotate(w, C), 500 + 1000 * rand(m, 1), 0.01 * randn(m, 2)], 1)

    if kind == "hemisphere":   # the nearest cameras of every camera, itself first, at least two degrees apart from it
        K = min(m, 4 * lmax)
        near = []
        for s in range(0, m, 2048):
            d = torch.cdist(C[s:s + 2048], C)
            d[(d > 0) & (d < 0.04 * radius)] = math.inf
            d[torch.arange(len(d), device=dev), torch.arange(s, s + len(d), device=dev)] = 0
            near.append(d.topk(K, dim=1, largest=False).indices)
        near = torch.cat(near)
        prob = torch.arange(2, lmax + 1, device=dev, dtype=torch.float64) ** -2.0
    pts, oc, op, count = [], [], [], 0
    while count < n:
        k = min(max(2 * (n - count), 1024), 40_000)
        if kind == "ring":
            X = 4 * rand(k, 3) - 2
            cand = torch.arange(m, device=dev).expand(k, m)
            L = torch.full((k,), m, device=dev)
        elif kind == "hemisphere":
            X = (10 * rand(k, 3) - 5) * (radius / 20.0)
            L = 2 + torch.multinomial(prob, k, replacement=True, generator=g)
            cand = near[torch.randint(m, (k,), generator=g, device=dev)]
        else:   # in front of a frame, tracked over L consecutive frames around it
            a = torch.randint(m, (k,), generator=g, device=dev)
            z = 4 + 26 * rand(k)
            px = (2 * rand(k, 2) - 1) * 0.8 * torch.tensor([HALF_W, HALF_H], dtype=torch.float64, device=dev)
            Y = torch.cat([px / true[a, 6:7] * z[:, None], z[:, None]], 1)
            X = _rotate(-true[a, :3], Y - true[a, 3:6])
            L = torch.randint(2, lmax + 1, (k,), generator=g, device=dev)
            first = a - (rand(k) * L).long()
            cand = (first[:, None] + torch.arange(lmax, device=dev)) % m
        uv, z = _pixels(true[cand], X[:, None, :].expand(-1, cand.shape[1], -1))
        ok = _inside(uv, z, 1.0 if kind == "drive" else 0.1)
        if kind == "ring":
            to_cam = C[None] - X[:, None]
            cosine = (X[:, None] * to_cam).sum(-1) / (X.norm(dim=1)[:, None] * to_cam.norm(dim=-1))
            ok &= cosine >= 0.5
        if kind == "drive":
            take = ok & (torch.arange(lmax, device=dev)[None] < L[:, None])
        else:
            take = ok & (ok.cumsum(1) <= L[:, None])
        sel = (take.sum(1) >= 2).nonzero()[: n - count, 0]
        rows, cols = take[sel].nonzero(as_tuple=True)
        pts.append(X[sel])
        oc.append(cand[sel][rows, cols])
        op.append(count + rows)
        count += len(sel)
    pts, oc, op = torch.cat(pts), torch.cat(oc), torch.cat(op)
    if case["entry"] == "adjoint":   # a fixed number of observations: the longest tracks are cut
        first = torch.cumsum(torch.bincount(op, minlength=n), 0) - torch.bincount(op, minlength=n)
        rank = torch.arange(len(op), device=dev) - first[op]
        keep = torch.argsort(rank, stable=True)[: 4 * n].sort().values
        oc, op = oc[keep], op[keep]
    order = torch.argsort(op * m + oc)
    oc, op = oc[order], op[order]
    uv = torch.cat([_pixels(true[oc[s:s + (1 << 20)]], pts[op[s:s + (1 << 20)]])[0] for s in range(0, len(oc), 1 << 20)])
    uv = uv + randn(len(oc), 2)
    if case["huber"] > 0:   # mismatched features
        bad = rand(len(oc)) < 0.03
        uv = torch.where(bad[:, None], uv + 5 * randn(len(oc), 2), uv)
    cams = true.clone()
    cams[:, :3] += 0.01 * randn(m, 3)
    cams[:, 3:6] = -_rotate(cams[:, :3], C) + 0.05 * randn(m, 3)
    pts0 = pts + 0.05 * randn(n, 3)
    return cams, pts0, oc.to(torch.int32), op.to(torch.int32), uv, C


def _spatial(C, cap, phase):
    """Wedges of at most cap cameras by azimuth."""
    m = len(C)
    l = max(1, math.ceil(m / cap))
    order = np.argsort(np.mod(np.arctan2(C[:, 1], C[:, 0]) - phase, 2 * np.pi), kind="stable")
    out = np.empty(m, np.int32)
    out[order] = np.arange(m) * l // m
    return out


def _joins(rng, m, pairs, cap):
    """Random joins of co-visible cameras up to cap cameras, small clusters first, as stochastic graph clustering
    makes them: about m / (0.8 cap) clusters of like sizes."""
    root, size = list(range(m)), [1] * m
    for limit in [max(2, cap // 16), max(2, cap // 8), max(2, cap // 4), cap // 2, cap]:
        for a, b in pairs[rng.integers(0, len(pairs), 8 * m)].tolist():
            while root[a] != a:
                root[a] = root[root[a]]
                a = root[a]
            while root[b] != b:
                root[b] = root[root[b]]
                b = root[b]
            if a != b and size[a] + size[b] <= limit:
                root[b] = a
                size[a] += size[b]
    for j in range(m):
        while root[j] != root[root[j]]:
            root[j] = root[root[j]]
    return np.unique(np.array(root), return_inverse=True)[1].astype(np.int32)


def _assignments(case, seed, oc, op, C):
    """The cluster assignment of every iteration, (iters, m) int32, or one (1, m) that is kept."""
    rng = np.random.default_rng([int(seed), case["cams"], 7])
    m, cap, C = case["cams"], case["cap"], C.cpu().numpy()
    if case["clusters"] == "uneven":
        sizes = []
        while sum(sizes) < m:
            sizes.append(min(int(rng.integers(20, cap + 1)), m - sum(sizes)))
        return np.repeat(np.arange(len(sizes)), sizes).astype(np.int32)[None]
    if case["clusters"] == "spatial":
        return _spatial(C, cap, rng.uniform(0, 2 * np.pi))[None]
    same = op[1:] == op[:-1]
    pairs = torch.stack([oc[:-1][same], oc[1:][same]], 1).cpu().numpy()
    return np.stack([_joins(rng, m, pairs, cap) for _ in range(max(1, case["iters"]))])


# ------------------------------------------------------------------------------------------------------
def prepare(case, seed):
    cams, pts, oc, op, uv, C = _problem(case, seed)
    s = dict(case=case, cams=cams, pts=pts)
    if case["entry"] == "cost":
        s.update(oc=oc, op=op, uv=uv, F=torch.zeros(1, dtype=torch.float64, device=cams.device))
        return s
    draws = _assignments(case, seed, oc, op, C)
    solver = {"clusters": stba.STBA_SOLVER_CLUSTERS, "pcg_full": stba.STBA_SOLVER_PCG_FULL,
              "pcg_clusters": stba.STBA_SOLVER_PCG_CLUSTERS}[case["solver"]]
    s.update(draws=draws, out_c=torch.empty_like(cams), out_p=torch.empty_like(pts))
    s["ctx"] = stba.stba_create(cams, pts, oc, op, uv, draws[0], huber_a=case["huber"], lambda0=case["lambda0"],
                                linear_solver=solver,
                                precision=stba.STBA_FP64 if case["precision"] == "fp64" else stba.STBA_MIXED)
    if case["entry"] == "adjoint":
        g = torch.Generator(device=cams.device)
        g.manual_seed(int(seed) + 77)
        # the gradient of a loss on the camera positions and the points
        s["g_c"] = torch.randn(cams.shape, generator=g, device=cams.device, dtype=torch.float64)
        s["g_c"][:, 6:] = 0
        s["g_p"] = torch.randn(pts.shape, generator=g, device=cams.device, dtype=torch.float64)
    return s


def run(s):
    case = s["case"]
    if case["entry"] == "cost":
        stba.stba_cost_noalloc(s["cams"], s["pts"], s["oc"], s["op"], s["uv"], s["F"])
        return {"F": s["F"]}
    ctx, draws = s["ctx"], s["draws"]
    # new estimates of a kept problem: damping, parameters, then the iterations
    stba.stba_set_state(ctx, case["lambda0"], 0.0, 0)
    stba.stba_set_params(ctx, s["cams"], s["pts"])
    if case["entry"] == "adjoint":
        stba.stba_record(ctx, case["iters"])
    for t in range(case["iters"]):
        if len(draws) > 1:
            stba.stba_set_clusters(ctx, draws[t])
        stba.stba_lm_iteration(ctx, want_info=False)
    real = torch.float64 if case["precision"] == "fp64" else torch.float32
    _, F, _ = stba.stba_get_state(ctx)
    stba.stba_get_params(ctx, s["out_c"], s["out_p"])
    out = {"F": F, "cameras": s["out_c"].to(real, copy=True), "points": s["out_p"].to(real, copy=True)}
    if case["entry"] == "adjoint":
        gq, gc, gp = stba.stba_adjoint(ctx, s["g_c"], s["g_p"])
        out.update(g_obs=gq.to(real), g_cameras=gc.to(real), g_points=gp.to(real))
    return out


def _shape(case):
    """Expected observations, virtual points and camera-pair instances per iteration of a case."""
    n, L = case["points"], case["lmax"]
    if case["scene"] == "ring":
        k = 0.22 * case["cams"]
        q, pairs = n * k, n * k * k / 2
    elif case["scene"] == "drive":
        q, pairs = n * L * 0.4, n * L * L * 0.12
    else:
        z = sum(i ** -2.0 for i in range(2, L + 1))
        q = n * sum(i ** -1.0 for i in range(2, L + 1)) / z
        pairs = n * sum((i - 1) / (2 * i) for i in range(2, L + 1)) / z
    inside = {"joins": 0.09, "spatial": 0.7, "uneven": 0.9}[case["clusters"]]
    return q, pairs * (1.0 if case["cap"] >= case["cams"] or case["solver"] == "pcg_full" else inside)


def work(case):
    """Per iteration: every observation (two indices and a pixel) and the parameters read once and the parameters
    written once; Jacobians, Schur terms, camera-pair blocks, the dense factorisations and two solves."""
    m, n = case["cams"], case["points"]
    q, pairs = _shape(case)
    r = 8 if case["precision"] == "fp64" else 4
    if case["entry"] == "cost":
        return {"bytes": q * (8 + 16) + (9 * m + 3 * n) * 8 + 8, "flops": 45 * q}
    byts = q * (8 + 2 * r) + 2 * (9 * m + 3 * n) * 8
    l = math.ceil(m / min(m, case["cap"] * (0.55 if case["clusters"] == "uneven" else 0.85 if case["clusters"] == "joins" else 1)))
    d = 9.0 * m / l
    flops = q * (300 + 350 + 100 + 45) + pairs * 2 * 243
    if case["solver"] == "clusters":
        flops += l * (d ** 3 / 3 + 8 * d * d)
    else:
        flops += 20 * q * 2 * (36 + 12)
    if case["entry"] == "adjoint":
        byts, flops = 3 * byts + q * 2 * 8, 2 * flops + q * 6 * 600
    return {"bytes": case["iters"] * byts, "flops": case["iters"] * flops}


# ------------------------------------------------------------------------------------------------------
# the same in plain torch, FP64
def _jacobians(c, X):
    """Pixels (q, 2) and their derivatives by the camera (q, 2, 9) and the point (q, 2, 3)."""
    w, t, f, k1, k2 = c[:, :3], c[:, 3:6], c[:, 6], c[:, 7], c[:, 8]
    s = (w * w).sum(1)
    th = s.sqrt()
    A, B = th.sin() / th, 2 * (th / 2).sin() ** 2 / s
    dA, dB = (th.cos() - A) / (2 * s), (A / 2 - B) / s   # by s = |w|^2
    wx, wd = torch.linalg.cross(w, X), (w * X).sum(1)
    u = w * wd[:, None] - s[:, None] * X
    Y = X + A[:, None] * wx + B[:, None] * u + t
    I = torch.eye(3, dtype=c.dtype, device=c.device)

    def hat(a):
        z = torch.zeros_like(a[:, 0])
        return torch.stack([torch.stack([z, -a[:, 2], a[:, 1]], 1), torch.stack([a[:, 2], z, -a[:, 0]], 1),
                            torch.stack([-a[:, 1], a[:, 0], z], 1)], 1)

    def outer(a, b):
        return a[:, :, None] * b[:, None, :]

    e3 = lambda v: v[:, None, None]   # noqa: E731
    R = I + e3(A) * hat(w) + e3(B) * (outer(w, w) - e3(s) * I)
    Yw = outer(2 * dA[:, None] * wx + 2 * dB[:, None] * u, w) - e3(A) * hat(X) + \
        e3(B) * (e3(wd) * I + outer(w, X) - 2 * outer(X, w))
    iz = 1 / Y[:, 2]
    x, y = Y[:, 0] * iz, Y[:, 1] * iz
    r2 = x * x + y * y
    d, de = 1 + r2 * (k1 + k2 * r2), 2 * (k1 + 2 * k2 * r2)
    xx, xy, yy = f * (d + de * x * x), f * de * x * y, f * (d + de * y * y)
    P = torch.stack([torch.stack([xx * iz, xy * iz, -(xx * x + xy * y) * iz], 1),
                     torch.stack([xy * iz, yy * iz, -(xy * x + yy * y) * iz], 1)], 1)
    xn = torch.stack([x, y], 1)
    inner = torch.stack([d, f * r2, f * r2 * r2], 1)
    return (f * d)[:, None] * xn, torch.cat([P @ Yw, P, xn[:, :, None] * inner[:, None, :]], 2), P @ R, Y[:, 2]


def _cost(cams, pts, oc, op, uv, a):
    F = torch.zeros((), dtype=torch.float64, device=cams.device)
    for s in range(0, len(oc), 1 << 21):
        pix, z = _pixels(cams[oc[s:s + (1 << 21)]], pts[op[s:s + (1 << 21)]])
        e = ((pix - uv[s:s + (1 << 21)]) ** 2).sum(1)
        if a > 0:
            e = torch.where(e <= a * a, e, 2 * a * e.sqrt() - a * a)
        F = F + e.sum() + (0.0 if bool((z > 1e-9).all()) else math.inf)
    return float(F)


def _step(cams, pts, oc, op, uv, cl, lam, a):
    """One damped, cluster-split Gauss-Newton step (dc, dp); every operation can be differentiated."""
    m, n, dev = len(cams), len(pts), cams.device

    def total(size, index, v):
        return torch.zeros((size,) + v.shape[1:], dtype=v.dtype, device=dev).index_add(0, index, v)

    pix, Jc, Jp, _ = _jacobians(cams[oc], pts[op])
    r = pix - uv
    if a > 0:
        e = (r * r).sum(1).sqrt()
        sw = torch.where(e <= a, torch.ones_like(e), (a / e).sqrt())
        r, Jc, Jp = r * sw[:, None], Jc * sw[:, None, None], Jp * sw[:, None, None]
    l = int(cl.max()) + 1
    vps, vp, cnt = torch.unique(op * l + cl[oc], return_inverse=True, return_counts=True)   # (point, cluster) copies
    vpt = vps // l
    JpT = Jp.transpose(1, 2)
    V, wv = total(len(vps), vp, JpT @ Jp), total(len(vps), vp, -(JpT @ r[:, :, None])[..., 0])
    Cp, wp = total(n, vpt, V), total(n, vpt, wv)
    if lam >= 0.1:   # steepest-descent correction: the copies of a point get one diagonal step
        wv = V.diagonal(dim1=1, dim2=2) * (wp / Cp.diagonal(dim1=1, dim2=2))[vpt]
    damp = lambda M: M + lam * torch.diag_embed(M.diagonal(dim1=1, dim2=2))   # noqa: E731
    Lv = torch.linalg.cholesky(damp(V))
    yv = torch.cholesky_solve(wv[:, :, None], Lv)
    # camera systems, dense per cluster in one flat buffer
    order = torch.argsort(cl, stable=True)
    sizes = torch.bincount(cl, minlength=l)
    start = torch.cumsum(sizes, 0) - sizes
    local = torch.empty_like(cl)
    local[order] = torch.arange(m, device=dev) - start[cl[order]]
    dim = 9 * sizes
    soff = torch.cumsum(dim * dim, 0) - dim * dim
    nine = torch.arange(9, device=dev)

    def where(i, j):   # flat indices of the 9 x 9 blocks of cameras i, j of one cluster
        k = cl[i]
        return (soff[k] + 9 * local[i] * dim[k] + 9 * local[j])[:, None, None] + nine[:, None] * dim[k][:, None, None] + nine

    G = torch.linalg.solve_triangular(Lv[vp], JpT @ Jc, upper=False)
    JcT = Jc.transpose(1, 2)
    D = total(m, oc, damp(JcT @ Jc) - G.transpose(1, 2) @ G)
    every = torch.arange(m, device=dev)
    S = torch.zeros(int((dim * dim).sum()), dtype=torch.float64, device=dev).index_add(0, where(every, every).reshape(-1), D.reshape(-1))
    by_vp = torch.argsort(vp, stable=True)
    rank = torch.arange(len(by_vp), device=dev) - (torch.cumsum(cnt, 0) - cnt)[vp[by_vp]]
    ends = torch.cumsum(rank, 0)
    for s0 in range(0, len(by_vp), 200_000):   # pairs (o, an earlier observation of the same copy)
        o, k = by_vp[s0:s0 + 200_000], rank[s0:s0 + 200_000]
        if int(k.sum()) == 0:
            continue
        pos = torch.repeat_interleave(torch.arange(s0, s0 + len(o), device=dev), k)
        back = torch.arange(len(pos), device=dev) - torch.repeat_interleave(torch.cumsum(k, 0) - k, k) + 1
        x, y = by_vp[pos], by_vp[pos - back]
        block = -(G[x].transpose(1, 2) @ G[y])
        S = S.index_add(0, where(oc[x], oc[y]).reshape(-1), block.reshape(-1))
        S = S.index_add(0, where(oc[y], oc[x]).reshape(-1), block.transpose(1, 2).reshape(-1))
    b = total(m, oc, -(JcT @ (r[:, :, None] + Jp @ yv[vp]))[..., 0])
    dc = torch.zeros_like(cams)
    for k in range(l):
        o, d = int(soff[k]), int(dim[k])
        mine = order[int(start[k]):int(start[k]) + int(sizes[k])]
        x = torch.cholesky_solve(b[mine].reshape(-1, 1), torch.linalg.cholesky(S[o:o + d * d].reshape(d, d)))
        dc = dc.index_add(0, mine, x.reshape(-1, 9))
    t = total(n, op, (JpT @ (Jc @ dc[oc][:, :, None]))[..., 0])
    dp = torch.linalg.solve(damp(Cp), (wp - t)[:, :, None])[..., 0]
    return dc, dp


def exact(case, seed):
    cams, pts, oc, op, uv, C = _problem(case, seed)
    oc, op = oc.long(), op.long()
    if case["entry"] == "cost":
        return {"F": torch.tensor([_cost(cams, pts, oc, op, uv, 0.0)], dtype=torch.float64)}
    draws = torch.from_numpy(_assignments(case, seed, oc, op, C)).to(cams.device).long()
    if case["solver"] == "pcg_full":
        draws = torch.zeros_like(draws)
    tape = case["entry"] == "adjoint"
    if tape:
        cams, pts, uv = (v.requires_grad_() for v in (cams, pts, uv))
    c, p, lam, F = cams, pts, case["lambda0"], None
    with torch.set_grad_enabled(tape):
        for t in range(case["iters"]):
            if F is None:
                F = _cost(c.detach(), p.detach(), oc, op, uv.detach(), case["huber"])
            dc, dp = _step(c, p, oc, op, uv, draws[t % len(draws)], lam, case["huber"])
            Fn = _cost((c + dc).detach(), (p + dp).detach(), oc, op, uv.detach(), case["huber"])
            if Fn < F:
                c, p, F, lam = c + dc, p + dp, Fn, lam / 3
            else:
                lam *= 3
    out = {"F": F, "cameras": c.detach(), "points": p.detach()}
    if tape:
        g = torch.Generator(device=c.device)
        g.manual_seed(int(seed) + 77)
        g_c = torch.randn(c.shape, generator=g, device=c.device, dtype=torch.float64)
        g_c[:, 6:] = 0
        g_p = torch.randn(p.shape, generator=g, device=c.device, dtype=torch.float64)
        gc, gp, gq = torch.autograd.grad([c, p], [cams, pts, uv], [g_c, g_p])
        out.update(g_obs=gq, g_cameras=gc, g_points=gp)
    return out
