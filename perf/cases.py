"""The work that programs built on this library have it do, as cases to time.

A program holds one `Context` and hands it CUDA tensors: blob positions and
forces (products with the mobility), bodies with their forces (solves), or
bodies alone (kinematics, preconditioner).  `listed()` names the usual calls
over their usual sizes, `draw()` gives others of the same ranges.

Kinds of case
  matvec      u = M f: `fp32` is the product of every Krylov step of a mixed-
              precision solve and of a time stepper, `fp64` the one of plain
              FP64 solves, `df64` the refinement residual's
  noalloc     the same product from a program that owns all device memory
  eval        velocity of tracers at points of the fluid (flow plots)
  kinematics  blob build, K and K^T once each: what a time step does besides
              the products
  precond     setup of the block-diagonal preconditioner for a configuration
              and one application
  solve       one mobility problem
  batch       several independent mobility problems in one call

The FP32 products are accurate to FP32 rounding (about 5e-7), so a program
that asks for them keeps them in FP32: `run` returns those as float32.
"""
import math

import numpy as np
import torch

import paper_1602_02170_gb300 as mb
from paper_1602_02170_gb300 import inputs

A42, A162, A_MIXED = 0.243, 0.12, 0.1625  # blob radii of the 42- and 162-blob shells, mixed bodies
TOL = {"fp64": 1e-10, "mixed": 1e-11}  # of the solves; a mixed solve refines


def listed():
    return [
        # one step's product for the 8-shell suspension: latency and launches
        {"name": "matvec_fp32_336", "kind": "matvec", "prec": "fp32", "n": 336, "body": 42, "wall": True},
        # an ordinary cloud of blobs, not a multiple of any tile
        {"name": "matvec_fp32_9003", "kind": "matvec", "prec": "fp32", "n": 9003, "body": 0, "wall": True},
        # the benchmark's product
        {"name": "matvec_fp32_65536", "kind": "matvec", "prec": "fp32", "n": 65536, "body": 0, "wall": True},
        # a step of a plain FP64 solve of 65 shells of 42 blobs
        {"name": "matvec_fp64_2730", "kind": "matvec", "prec": "fp64", "n": 2730, "body": 42, "wall": True},
        # a refinement residual of 124 shells of 162 blobs
        {"name": "matvec_df64_20088", "kind": "matvec", "prec": "df64", "n": 20088, "body": 162, "wall": True},
        # product in an unbounded domain for a program that allocates nothing
        {"name": "noalloc_20011_free", "kind": "noalloc", "n": 20011, "body": 0, "wall": False},
        # flow in a plane of 64 x 48 points around 160 shells of 42 blobs
        {"name": "eval_fp32_3072x6720", "kind": "eval", "prec": "fp32", "points": 3072, "n": 6720, "wall": True},
        # the monolayer's blob build, K and K^T (663,552 blobs)
        {"name": "kinematics_4096x162", "kind": "kinematics", "bodies": 4096, "body": 162},
        # preconditioner of 300 shells and boomerangs
        {"name": "precond_300_mixed", "kind": "precond", "bodies": 300, "wall": True},
        # the plain FP64 mobility solve of 8 shells
        {"name": "solve_fp64_8x42", "kind": "solve", "prec": "fp64", "bodies": 8, "body": 42, "wall": True},
        # a monolayer patch in mixed precision
        {"name": "solve_mixed_256x162", "kind": "solve", "prec": "mixed", "bodies": 256, "body": 162, "wall": True},
        # suspensions of 8 to 100 bodies of two shapes in one call
        {"name": "batch_12_mixed", "kind": "batch", "problems": 12, "lo": 8, "hi": 100},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matvec"] * 5 + ["noalloc", "eval", "eval", "kinematics", "precond", "solve", "solve", "batch"])
    wall = rng.random() < 0.75
    if kind == "matvec":
        prec = rng.choice(["fp32", "fp32", "fp64", "df64"])
        body = rng.choice([0, 42, 162])
        n = _log(rng, 100, {"fp32": 65536, "fp64": 16384, "df64": 32768}[prec])
        return {"kind": kind, "prec": prec, "n": max(1, n // body) * body if body else n, "body": body, "wall": wall}
    if kind == "noalloc":
        return {"kind": kind, "n": _log(rng, 100, 65536), "body": 0, "wall": wall}
    if kind == "eval":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        top = 30000 if prec == "fp32" else 6000
        return {"kind": kind, "prec": prec, "points": _log(rng, 16, top), "n": 42 * _log(rng, 1, top // 42), "wall": wall}
    if kind == "kinematics":
        return {"kind": kind, "bodies": _log(rng, 8, 4096), "body": rng.choice([12, 42, 162])}
    if kind == "precond":
        return {"kind": kind, "bodies": _log(rng, 8, 400), "wall": wall}
    if kind == "solve":
        prec = rng.choice(["fp64", "mixed", "mixed"])
        body = rng.choice([12, 42, 162])
        top = 2500 if prec == "fp64" else 40000
        return {"kind": kind, "prec": prec, "bodies": _log(rng, 4, min(256, top // body)), "body": body, "wall": wall}
    lo = _log(rng, 8, 20)
    return {"kind": kind, "problems": rng.randint(2, 12), "lo": lo, "hi": lo * rng.randint(2, 5)}


# ---------------------------------------------------------------- inputs
_context = None


def _ctx():
    """The context that a program keeps for as long as it runs."""
    global _context
    if _context is None:
        _context = mb.Context(0)
    return _context


def _dev(x):
    x = np.ascontiguousarray(x)
    return torch.as_tensor(x).to("cuda", torch.int64 if x.dtype == np.int64 else torch.float64)


def _radius(body):
    return {0: 0.5, 12: 0.5, 42: A42, 162: A162}[body]


def _shells(rng, n_bodies, body):
    """Shells in a layer above the wall, at the monolayer's density (one per
    3.125 x 3.125): a square lattice, each centre moved about in its cell."""
    a = _radius(body)
    side = math.ceil(math.sqrt(n_bodies))
    gap = max(0.0, 3.125 - 2.0 * (1.0 + a))
    at = rng.permutation(side * side)[:n_bodies]
    q = np.empty((n_bodies, 3))
    q[:, 0] = (at % side + 0.5) * 3.125 + rng.uniform(-0.5, 0.5, n_bodies) * gap
    q[:, 1] = (at // side + 0.5) * 3.125 + rng.uniform(-0.5, 0.5, n_bodies) * gap
    q[:, 2] = rng.uniform(1.05 + a, 1.45 + a, n_bodies)
    theta = inputs.random_unit_quaternions(rng, n_bodies)
    F = rng.normal(0.0, 0.1, (n_bodies, 3))
    F[:, 2] -= 1.0
    T = rng.normal(0.0, 0.1, (n_bodies, 3))
    start = np.arange(n_bodies + 1, dtype=np.int64) * body
    return {"q": _dev(q), "theta": _dev(theta), "blob_start": _dev(start),
            "rho": _dev(np.tile(inputs.shell(body), (n_bodies, 1))), "F": _dev(F), "T": _dev(T)}


def _mixed(rng, n_bodies):
    """42-blob shells and 15-blob boomerangs in turn, at the density of the
    library's mixed suspensions (one per 5 x 5), every blob above the wall."""
    side = math.ceil(math.sqrt(n_bodies))
    at = rng.permutation(side * side)[:n_bodies]
    shapes = [inputs.shell(42), inputs.boomerang15()]
    reach = np.array([np.linalg.norm(s, axis=1).max() for s in shapes])[np.arange(n_bodies) % 2]
    gap = 5.0 - 2.0 * (1.65 + A_MIXED)
    q = np.empty((n_bodies, 3))
    q[:, 0] = (at % side + 0.5) * 5.0 + rng.uniform(-0.5, 0.5, n_bodies) * gap
    q[:, 1] = (at // side + 0.5) * 5.0 + rng.uniform(-0.5, 0.5, n_bodies) * gap
    q[:, 2] = rng.uniform(reach + 1.05 * A_MIXED, 3.0)
    count = np.array([len(s) for s in shapes])[np.arange(n_bodies) % 2]
    F = rng.normal(0.0, 0.1, (n_bodies, 3))
    F[:, 2] -= 1.0
    return {"q": _dev(q), "theta": _dev(inputs.random_unit_quaternions(rng, n_bodies)),
            "blob_start": _dev(np.concatenate([[0], np.cumsum(count)]).astype(np.int64)),
            "rho": _dev(np.concatenate([shapes[p % 2] for p in range(n_bodies)])),
            "F": _dev(F), "T": _dev(rng.normal(0.0, 0.1, (n_bodies, 3)))}


def _blobs(rng, n, body):
    """n blob positions: a cloud at the benchmark's density, or shells."""
    if not body:
        side = 400.0 * math.sqrt(n / 65536.0)
        a = _radius(0)
        return _dev(np.stack([rng.uniform(0, side, n), rng.uniform(0, side, n), rng.uniform(a, 3 * a, n)], axis=1))
    return _positions(_shells(rng, n // body, body))


def _counts(case):
    """Bodies of each problem of a batch, spread evenly over the logarithm."""
    return [int(round(case["lo"] * (case["hi"] / case["lo"]) ** (k / (case["problems"] - 1))))
            for k in range(case["problems"])]


def _inputs(case, seed):
    rng = np.random.default_rng([seed, 1602])
    kind = case["kind"]
    if kind in ("matvec", "noalloc"):
        return {"r": _blobs(rng, case["n"], case["body"]), "f": _dev(rng.standard_normal((case["n"], 3))),
                "a": _radius(case["body"])}
    if kind == "eval":
        r = _blobs(rng, case["n"], 42)
        side = 3.125 * math.ceil(math.sqrt(case["n"] // 42))
        x = np.stack([rng.uniform(0, side, case["points"]), np.full(case["points"], 0.5 * side),
                      rng.uniform(A42, 4.0, case["points"])], axis=1)
        return {"r": r, "x": _dev(x), "f": _dev(rng.standard_normal((case["n"], 3))), "a": A42}
    if kind == "kinematics":
        n = case["bodies"] * case["body"]
        return dict(_shells(rng, case["bodies"], case["body"]), UO=_dev(rng.standard_normal((case["bodies"], 6))),
                    lam=_dev(rng.standard_normal((n, 3))))
    if kind == "precond":
        s = _mixed(rng, case["bodies"])
        return dict(s, r=_positions(s), w=_dev(rng.standard_normal(tuple(s["rho"].shape))),
                    g=_dev(rng.standard_normal((case["bodies"], 6))), a=A_MIXED)
    if kind == "solve":
        return dict(_shells(rng, case["bodies"], case["body"]), a=_radius(case["body"]))
    return {"problems": [_mixed(rng, c) for c in _counts(case)], "a": A_MIXED}


def prepare(case, seed):
    return dict(_inputs(case, seed), case=case, ctx=_ctx())


# ---------------------------------------------------------------- the calls
def run(state):
    c, ctx = state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "matvec":
        u = ctx.mobility_matvec(state["r"], state["f"], state["a"], 1.0, c["wall"], c["prec"])
        return u.to(torch.float32) if c["prec"] == "fp32" else u
    if kind == "noalloc":
        return mb.mobility_matvec_noalloc(state["r"], state["f"], state["a"], 1.0, c["wall"]).to(torch.float32)
    if kind == "eval":
        u = ctx.mobility_eval(state["x"], state["r"], state["f"], state["a"], 1.0, c["wall"], c["prec"])
        return u.to(torch.float32) if c["prec"] == "fp32" else u
    if kind == "kinematics":
        r = ctx.blob_positions(state["q"], state["theta"], state["blob_start"], state["rho"])
        return {"r": r, "v": ctx.K_apply(r, state["q"], state["blob_start"], state["UO"]),
                "FT": ctx.KT_apply(r, state["q"], state["blob_start"], state["lam"])}
    if kind == "precond":
        ctx.precond_setup(state["r"], state["q"], state["blob_start"], state["a"], 1.0, c["wall"])
        lam, UO = ctx.precond_apply(state["w"], state["g"])
        return {"lam": lam, "UO": UO}
    if kind == "solve":
        U, Om, lam, _ = ctx.solve_mobility(state["q"], state["theta"], state["blob_start"], state["rho"], state["F"],
                                           state["T"], state["a"], 1.0, c["wall"], tol=TOL[c["prec"]], prec=c["prec"])
        return {"U": U, "Omega": Om, "lam": lam}
    return [{"U": U, "Omega": Om, "lam": lam}
            for U, Om, lam, _ in ctx.solve_batch(state["problems"], state["a"], 1.0, True, tol=TOL["mixed"], prec="mixed")]


def work(case):
    """108 operations per ordered pair with the wall and 29 without (the
    formula of the mobility as written), products of a solve at 16 steps,
    one Cholesky and one assembly per body for the preconditioner."""
    kind = case["kind"]
    pair = 108 if case.get("wall", True) else 29
    if kind in ("matvec", "noalloc"):
        return {"bytes": 72 * case["n"], "flops": pair * case["n"] ** 2}
    if kind == "eval":
        return {"bytes": 48 * (case["n"] + case["points"]), "flops": pair * case["n"] * case["points"]}
    if kind == "kinematics":
        blobs = case["bodies"] * case["body"]
        return {"bytes": 144 * blobs + 250 * case["bodies"], "flops": 66 * blobs}

    def body(n):
        return (3 * n) ** 3 / 3 + pair * n * n / 2

    if kind == "solve":
        problems = [(case["bodies"], case["bodies"] * case["body"], case["bodies"] * body(case["body"]))]
    else:
        problems = [(c, 42 * ((c + 1) // 2) + 15 * (c // 2), (c + 1) // 2 * body(42) + c // 2 * body(15))
                    for c in ([case["bodies"]] if kind == "precond" else _counts(case))]
    if kind == "precond":
        return {"bytes": sum(96 * n + 150 * c for c, n, _ in problems), "flops": sum(b for _, _, b in problems)}
    return {"bytes": sum(48 * n + 200 * c for c, n, _ in problems),
            "flops": sum(b + 16 * pair * n * n for _, n, b in problems)}


# ---------------------------------------------------------------- in 64 bits
def _positions(s):
    """q + R(theta) rho, quaternions scalar first."""
    count = s["blob_start"][1:] - s["blob_start"][:-1]
    of = torch.repeat_interleave(torch.arange(len(count), device=count.device), count)
    th = (s["theta"] / s["theta"].norm(dim=1, keepdim=True))[of]
    w, v = th[:, :1], th[:, 1:]
    t = 2.0 * torch.linalg.cross(v, s["rho"])
    return (s["q"][of] + s["rho"] + w * t + torch.linalg.cross(v, t)).contiguous()


def _pairs(x, y, a, wall):
    """The nine entries of M(x_t, y_j), unit viscosity, each (targets, sources).

    Rotne-Prager-Yamakawa with the overlap form below 2a; with the wall, the
    image part of Blake's tensor with (1 + a^2/6 Laplacian) at both points:
    for R = x - (y with z reflected), e = R/|R|, hs, ht = heights / |R|."""
    dx, dy, dz = (x[:, None, k] - y[None, :, k] for k in range(3))
    dxy2 = dx * dx + dy * dy
    r = (dxy2 + dz * dz).sqrt()
    near = r < 2 * a
    ri = 1.0 / r.clamp_min(1e-150)
    C = torch.where(near, 1 - 9 * r / (32 * a), 0.75 * a * ri + 0.5 * (a * ri) ** 3)
    D = torch.where(near, 3 / (32 * a) * ri, (0.75 * a * ri - 1.5 * (a * ri) ** 3) * ri * ri)
    d = (dx, dy, dz)
    M = {(p, q): D * d[p] * d[q] for p in range(3) for q in range(3)}
    for p in range(3):
        M[p, p] = M[p, p] + C
    del r, ri, near, C, D
    if wall:
        zt, zs = x[:, None, 2], y[None, :, 2]
        R3 = zt + zs
        inv = (dxy2 + R3 * R3).rsqrt()
        hs, ht = zs * inv, zt * inv
        e3 = hs + ht
        E, p, X = e3 * e3, hs * ht, (a * inv) ** 2
        f1 = -1 - 2 * p + X * (2 * E - 2 / 3) + X * X * (2 / 3 - 10 / 3 * E)
        f2 = -1 + 6 * p + X * (2 - 10 * E) + X * X * (70 / 3 * E - 10 / 3)
        f3 = 2 * hs + e3 * (X * (20 * E - 4) + X * X * (40 / 3 - 140 / 3 * E) - 12 * p)
        f4 = 2 * hs - 20 / 3 * e3 * X * X
        f5 = -4 * hs * hs - 4 * E * X + X * X * (20 * E - 8 / 3)
        s = 0.75 * a * inv
        e = (dx * inv, dy * inv, e3)
        for i in range(3):
            for j in range(3):
                W = f2 * e[i] * e[j]
                if i == j:
                    W = W + f1
                if j == 2:
                    W = W + f3 * e[i]
                if i == 2:
                    W = W + f4 * e[j]
                if i == j == 2:
                    W = W + f5
                M[i, j] = M[i, j] + s * W
    scale = 1.0 / (6.0 * math.pi * a)
    return {k: scale * v for k, v in M.items()}


def _product(x, y, f, a, wall):
    step = max(1, (1 << 24) // len(y))
    out = []
    for b in range(0, len(x), step):
        M = _pairs(x[b:b + step], y, a, wall)
        out.append(torch.stack([sum(M[i, j] @ f[:, j] for j in range(3)) for i in range(3)], dim=1))
    return torch.cat(out)


def _dense(r, a, wall):
    n = len(r)
    M = torch.empty((n, 3, n, 3), dtype=torch.float64, device=r.device)
    step = max(1, (1 << 24) // n)
    for b in range(0, n, step):
        for (i, j), v in _pairs(r[b:b + step], r, a, wall).items():
            M[b:b + step, i, :, j] = v
    return M.view(3 * n, 3 * n)


def _K(r, q, start):
    """The (3N, 6 n_b) matrix of v_i = U_p + Omega_p x (r_i - q_p)."""
    count = start[1:] - start[:-1]
    of = torch.repeat_interleave(torch.arange(len(count), device=count.device), count)
    n = torch.arange(len(r), device=r.device)
    d = r - q[of]
    K = torch.zeros((len(r), 3, len(q), 6), dtype=torch.float64, device=r.device)
    for k in range(3):
        K[n, k, of, k] = 1.0
    for k, (u, v) in enumerate(((1, 2), (2, 0), (0, 1))):  # (Omega x d)_k = Omega_u d_v - Omega_v d_u
        K[n, k, of, 3 + u] = d[:, v]
        K[n, k, of, 3 + v] = -d[:, u]
    return K.view(3 * len(r), 6 * len(q))


def _saddle(M, K, w, g):
    """[[M, -K], [-K^T, 0]] [lam; U] = [w; g] by the Schur complement."""
    L = torch.linalg.cholesky(M)
    G = torch.linalg.solve_triangular(L, torch.cat([K, w[:, None]], dim=1), upper=False)
    G, y = G[:, :-1], G[:, -1:]
    U = torch.linalg.solve(G.T @ G, -g[:, None] - G.T @ y)
    lam = torch.linalg.solve_triangular(L.T, y + G @ U, upper=True)
    return lam.view(-1, 3), U.view(-1, 6)


def _mobility(s, a, wall):
    r = _positions(s)
    w = torch.zeros(3 * len(r), dtype=torch.float64, device=r.device)
    g = -torch.cat([s["F"], s["T"]], dim=1).reshape(-1)
    lam, U = _saddle(_dense(r, a, wall), _K(r, s["q"], s["blob_start"]), w, g)
    return {"U": U[:, :3].contiguous(), "Omega": U[:, 3:].contiguous(), "lam": lam}


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind in ("matvec", "noalloc"):
        return _product(s["r"], s["r"], s["f"], s["a"], case["wall"])
    if kind == "eval":
        return _product(s["x"], s["r"], s["f"], s["a"], case["wall"])
    if kind == "kinematics":
        r = _positions(s)
        nb, per = case["bodies"], case["body"]
        d = (r.view(nb, per, 3) - s["q"][:, None])
        lam = s["lam"].view(nb, per, 3)
        v = s["UO"][:, None, :3] + torch.linalg.cross(s["UO"][:, None, 3:].expand(nb, per, 3), d)
        return {"r": r, "v": v.reshape(-1, 3),
                "FT": torch.cat([lam.sum(1), torch.linalg.cross(d, lam).sum(1)], dim=1)}
    if kind == "precond":
        lam, UO = torch.empty_like(s["w"]), torch.empty_like(s["g"])
        start = s["blob_start"].tolist()
        for p in range(case["bodies"]):
            b = slice(start[p], start[p + 1])
            one = torch.tensor([0, start[p + 1] - start[p]], device="cuda")
            lam[b], UO[p:p + 1] = _saddle(_dense(s["r"][b], s["a"], case["wall"]),
                                          _K(s["r"][b], s["q"][p:p + 1], one), s["w"][b].reshape(-1), s["g"][p])
        return {"lam": lam, "UO": UO}
    if kind == "solve":
        return _mobility(s, s["a"], case["wall"]) if case["bodies"] * case["body"] <= 8000 else None
    return [_mobility(p, s["a"], True) for p in s["problems"]]
