"""Performance cases: what a program asks of this framework, through its
public Python entry points, from the smallest solves to the largest meshes.

Every case solves the 2D TM Maxwell system on a seeded jittered triangle mesh.
``prepare`` sets up what the program keeps (solvers, fields, a batch or a
server), ``run`` is one pass, ``work`` the bytes and operations the pass
cannot do without, ``exact`` the result in 64 bits by a plain torch
implementation of the method that shares no code with the framework.
"""
import math

import numpy as np
import torch

import paper_1304_5546_gb300 as P

L2_BYTES = 129e6
SPEEDS = (0.5, 1.0, 2.0)  # wave speeds of a medium's elements


def listed():
    return [
        # the plain method at its smallest: an FP64 cavity solve, 128
        # elements, from t = 0 to t = 1; launches and latency
        {"name": "cavity_f64_n4", "kind": "solve", "N": 4, "nx": 8, "ny": 8, "box": 2.0, "T": 1.0,
         "precision": "fp64"},
        # one served request solved on its own, at the small end of their
        # sizes: a point source on a mesh of about a thousand elements
        {"name": "source_n3", "kind": "source", "N": 3, "nx": 23, "ny": 23, "steps": 48,
         "precision": "fp32"},
        # right-hand sides for a caller's own integrator, in a medium, on a
        # mesh that stays in L2
        {"name": "rhs_media_n4", "kind": "rhs", "N": 4, "nx": 101, "ny": 101, "media": True,
         "odd": True, "precision": "fp32"},
        # an ordinary mesh at a high order
        {"name": "step_n6", "kind": "step", "N": 6, "nx": 161, "ny": 161, "steps": 4,
         "precision": "fp32"},
        # the benchmark's mesh and order
        {"name": "step_n5_large", "kind": "step", "N": 5, "nx": 707, "ny": 707, "steps": 4,
         "precision": "fp32"},
        # the order sweep at its low end: about 1e7 nodal values per field
        {"name": "step_n2_large", "kind": "step", "N": 2, "nx": 913, "ny": 913, "steps": 4,
         "precision": "fp32"},
        # the precision path: its mesh and order with FP32-accurate products,
        # and the split BF16 products on a ragged smaller one
        {"name": "step_n7_large", "kind": "step", "N": 7, "nx": 362, "ny": 362, "steps": 2,
         "precision": "fp32"},
        {"name": "step_n7_bf16x3", "kind": "step", "N": 7, "nx": 173, "ny": 144, "steps": 5,
         "odd": True, "precision": "bf16x3"},
        # an FP64 run of the kind FP32 results are judged by
        {"name": "step_n5_f64", "kind": "step", "N": 5, "nx": 225, "ny": 225, "steps": 1,
         "precision": "fp64"},
        # field sets that live in host memory: copied in, stepped, copied out
        {"name": "host_jobs_n5", "kind": "jobs", "N": 5, "nx": 354, "ny": 354, "jobs": 4,
         "steps": 1, "precision": "fp32"},
        # many problems of uneven size and mixed order stepped together
        {"name": "batch_n357", "kind": "batch", "problems": 24, "k_lo": 500, "k_hi": 50000,
         "orders": "3,5,7", "steps": 20},
        # requests solved by the continuous-batching server
        {"name": "server_n3to7", "kind": "server", "problems": 20, "k_lo": 1000, "k_hi": 20000,
         "orders": "3,4,5,6,7", "steps": 48},
    ]


def _spread(rng, lo, hi):
    """An integer of [lo, hi], uniform in its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "rhs", "rhs", "solve", "source", "jobs",
                       "batch", "server"])
    if kind in ("batch", "server"):
        lo, hi = (500, 50000) if kind == "batch" else (1000, 20000)
        orders = sorted(rng.sample(range(1, 8) if kind == "batch" else range(3, 8),
                                   rng.randint(2, 4)))
        return {"kind": kind, "problems": rng.randint(3, 24 if kind == "batch" else 20),
                "k_lo": lo, "k_hi": _spread(rng, 4 * lo, hi),
                "orders": ",".join(str(n) for n in orders), "steps": rng.randint(3, 16)}
    N = rng.randint(1, 7)
    Np = (N + 1) * (N + 2) // 2
    fp64 = kind in ("step", "rhs", "solve") and rng.random() < 0.25
    most = {"step": 1.8e7, "rhs": 1.8e7, "solve": 4e4, "source": 4e5, "jobs": 4e6}[kind]
    if fp64:
        most = min(most, 1.8e6)
    K = _spread(rng, 128, max(256, int(most / Np)))
    shape = math.sqrt(rng.uniform(0.5, 2.0))
    nx = max(2, int(math.sqrt(K / 2) * shape))
    ny = max(2, int(K / 2 / nx))
    case = {"kind": kind, "N": N, "nx": nx, "ny": ny, "odd": rng.random() < 0.5,
            "media": rng.random() < 0.3, "precision": "fp64" if fp64 else "fp32"}
    if kind in ("step", "rhs") and not fp64 and not case["media"]:
        case["precision"] = rng.choice(["fp32"] * 6 + ["tf32", "bf16", "bf16x3"])
    nodes = 2 * nx * ny * Np
    if kind == "solve":
        case.update(box=2.0, T=0.1)
    elif kind == "source":
        case["steps"] = rng.randint(5, 60)
    elif kind == "step":
        case["steps"] = 1 if fp64 else rng.randint(1, max(1, min(40, int(4e7 / nodes))))
    elif kind == "jobs":
        case.update(jobs=rng.randint(1, 4), steps=1)
    return case


# ------------------------------------------------------------------ inputs
def _mesh(nx, ny, rng, odd=False, box=1.0, jitter=0.3):
    """A jittered nx x ny grid of the given width, each square cut along its
    Delaunay diagonal, triangles counter-clockwise and listed square by
    square.  odd: without the last triangle."""
    h = box / max(nx, ny)
    gx, gy = np.meshgrid(np.arange(nx + 1) * h, np.arange(ny + 1) * h)
    dx = rng.uniform(-jitter * h, jitter * h, gx.shape)
    dy = rng.uniform(-jitter * h, jitter * h, gy.shape)
    dx[:, [0, -1]] = 0.0
    dy[[0, -1], :] = 0.0
    x, y = (gx + dx).ravel(), (gy + dy).ravel()
    a = (np.arange(ny)[:, None] * (nx + 1) + np.arange(nx)[None, :]).ravel()
    b, c, d = a + 1, a + nx + 2, a + nx + 1

    def angle(at, p, q):
        ux, uy, vx, vy = x[p] - x[at], y[p] - y[at], x[q] - x[at], y[q] - y[at]
        return np.arctan2(ux * vy - uy * vx, ux * vx + uy * vy) % (2 * np.pi)

    ac = angle(b, c, a) + angle(d, a, c) <= np.pi
    E = np.empty((2 * nx * ny, 3), np.int32)
    E[0::2] = np.stack([a, b, np.where(ac, c, d)], 1)
    E[1::2] = np.stack([np.where(ac, a, b), c, d], 1)
    if odd:
        E = E[:-1]
        used, E = np.unique(E, return_inverse=True)
        x, y, E = x[used], y[used], E.reshape(-1, 3).astype(np.int32)
    return x, y, E


def _eps(K, rng):
    return 1.0 / np.asarray(SPEEDS)[rng.integers(0, len(SPEEDS), K)] ** 2


def _pulse(x, y, centre, width):
    """Gaussian Ez, no H."""
    ez = torch.exp(-((x - centre[0]) ** 2 + (y - centre[1]) ** 2) / width ** 2)
    return torch.stack([torch.zeros_like(ez), torch.zeros_like(ez), ez])


def _problem(case, seed):
    """Mesh, permittivity, initial field and source of a single-mesh case."""
    rng = np.random.default_rng(seed)
    box = case.get("box", 1.0)
    V = _mesh(case["nx"], case["ny"], rng, case.get("odd", False), box)
    eps = _eps(len(V[2]), rng) if case.get("media") else None
    span = (V[0].max(), V[1].max())
    centre = [float(rng.uniform(0.3, 0.7)) * s for s in span]
    return {"mesh": V, "N": case["N"], "eps": eps, "centre": centre, "width": 0.1 * box,
            "rng": rng}


def _sizes(case):
    """(order, element count) of every problem: counts log-uniform."""
    rng = np.random.default_rng(case["problems"])
    orders = [int(n) for n in case["orders"].split(",")]
    k = np.exp(rng.uniform(math.log(case["k_lo"]), math.log(case["k_hi"]), case["problems"]))
    return [(orders[i % len(orders)], float(v)) for i, v in enumerate(k)]


def _problems(case, seed):
    """The problems of a batch or the requests of a server; their sizes are
    the case's own, the rest comes from the seed."""
    rng = np.random.default_rng(seed)
    got = []
    for N, K in _sizes(case):
        n = max(2, int(round(math.sqrt(K / 2))))
        V = _mesh(n, n, rng)
        p = {"mesh": V, "N": N, "eps": None,
             "centre": rng.uniform(0.3, 0.7, 2).tolist(), "width": 0.1}
        if case["kind"] == "batch":
            p["eps"] = _eps(len(V[2]), rng)
        got.append(p)
    return got


def _fields(p, xy, dtype):
    x, y = (torch.as_tensor(v).cuda() for v in xy)
    return _pulse(x, y, p["centre"], p["width"]).to(dtype)


def _edge_nodes(N):
    """Legendre-Gauss-Lobatto nodes."""
    inner = np.polynomial.legendre.Legendre.basis(N).deriv().roots()
    return np.concatenate([[-1.0], np.sort(inner.real), [1.0]])


def _cfl_dt(p):
    """The time step rule of the framework (dg_cfl_dt)."""
    x, y, E = p["mesh"]
    X, Y = x[E], y[E]
    ex, ey = np.roll(X, -1, 1) - X, np.roll(Y, -1, 1) - Y
    area2 = ex[:, 0] * ey[:, 1] - ey[:, 0] * ex[:, 1]
    rad = area2 / np.hypot(ex, ey).sum(1)
    if p["eps"] is not None:
        rad = rad * np.sqrt(p["eps"])
    g = _edge_nodes(p["N"])
    return 2.0 / 3.0 * float(rad.min()) * float(g[1] - g[0])


def _ricker_of(p, dt, steps):
    """A Ricker source whose peak falls into the solve: x, y, f, t0, amplitude."""
    f = 2.4 / (dt * steps)
    return (p["centre"][0], p["centre"][1], f, 1.2 / f, 1.0)


def _solver(p, precision="fp32"):
    return P.Solver(*p["mesh"], p["N"], precision=precision, eps=p["eps"])


# -------------------------------------------------------------------- pass
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "server"):
        todo = _problems(case, seed)
        cap = {}
        for p in todo:
            cap[p["N"]] = cap.get(p["N"], 0) + (len(p["mesh"][2]) + 3) // 4 * 4 + 4
        if kind == "server":
            s = {"kind": kind, "server": P.Server(cap), "requests": []}
            for p in todo:
                op = _solver(p)
                dt = _cfl_dt(p)
                out = np.empty((3, op.K, op.Np), np.float32)
                s["requests"].append((op, dt * (case["steps"] - 0.5),
                                      _ricker_of(p, dt, case["steps"]), out))
            return s
        s = {"kind": kind, "batch": P.Batch(cap), "steps": case["steps"], "slots": []}
        for p in todo:
            op = _solver(p)
            slot = s["batch"].add(op, _cfl_dt(p))
            q = _fields(p, op.nodes(), torch.float32).contiguous()
            P.dg_batch_set_fields(s["batch"].batch, slot, q, op.K * op.Np)
            s["slots"].append((slot, q, op.K * op.Np, op))
        torch.cuda.synchronize()
        return s
    p = _problem(case, seed)
    op = _solver(p, case["precision"])
    s = {"kind": kind, "op": op, "dt": _cfl_dt(p), "steps": case.get("steps", 0)}
    if kind == "source":
        P.dg_operator_set_source(op.op, _ricker_of(p, s["dt"], s["steps"]))
        s.update(q=op.new_fields(), res=op.new_fields(), T=s["dt"] * (s["steps"] - 0.5))
        return s
    q0 = _fields(p, op.nodes(), op.dtype)
    if kind == "jobs":
        s["host"] = []
        for j in range(case["jobs"]):
            h = torch.zeros((3, op.fstride), dtype=op.dtype, pin_memory=True)
            op.view(h).copy_((q0 / (j + 1)).cpu())
            s["host"].append(h)
        s["work"] = torch.empty(P.dg_step_host_jobs_work_bytes(op.op), dtype=torch.uint8,
                                device="cuda")
        return s
    s.update(q=op.new_fields(), res=op.new_fields())
    op.view(s["q"]).copy_(q0)
    if kind == "solve":
        s.update(T=case["T"], q0=s["q"].clone())
    return s


def run(s):
    kind = s["kind"]
    if kind == "server":
        srv = s["server"]
        ids = [srv.submit(op, T, source=src, out=out) for op, T, src, out in s["requests"]]
        for i in ids:
            srv.wait(i)
            srv.release(i)
        return [out for _, _, _, out in s["requests"]]
    if kind == "batch":
        s["batch"].step(s["steps"])
        for slot, q, stride, _ in s["slots"]:
            P.dg_batch_get_fields(s["batch"].batch, slot, q, stride)
        return [q for _, q, _, _ in s["slots"]]
    op = s["op"]
    if kind == "rhs":
        return op.view(op.rhs(s["q"], out=s["res"]))
    if kind == "step":
        op.step(s["q"], s["res"], s["dt"], s["steps"])
    elif kind == "solve":
        s["q"].copy_(s["q0"])
        op.solve(s["q"], s["res"], s["T"])
    elif kind == "source":
        s["q"].zero_()
        op.solve(s["q"], s["res"], s["T"])
    elif kind == "jobs":
        P.dg_step_host_jobs(op.op, s["host"], s["work"], 0.0, s["dt"], s["steps"])
        return [op.view(h) for h in s["host"]]
    return op.view(s["q"])


# -------------------------------------------------------------------- work
def _work_of(N, K, stages, size, media=False, rhs=False):
    """Bytes and operations of `stages` stages of one problem.  A working set
    beyond L2 passes through device memory once per stage (fields in and out,
    residual in and out except into a step's first stage, records and face
    codes in); a smaller one once in all.  Operations: 6 reference-axis
    products, chain rule, 3 lifts and fluxes of a right-hand side, and 5 per
    value for the update."""
    Np, Nafp = (N + 1) * (N + 2) // 2, 3 * (N + 1)
    fields = 3 * Np * size
    fixed = (20 if media else 13) * size + 12
    flops = 12 * Np * Np + 26 * Np + 3 * (2 * Np * Nafp + Np) + 18 * Nafp
    if rhs:
        return {"bytes": K * (2 * fields + fixed), "flops": K * flops}
    if K * (3 * fields + fixed) <= L2_BYTES:
        total = 2 * fields + fixed
    else:
        total = stages / 5 * (19 * fields + 5 * fixed)
    return {"bytes": K * total, "flops": K * stages * (flops + 5 * 3 * Np)}


def work(case):
    if case["kind"] in ("batch", "server"):
        parts = [_work_of(N, K, 5 * case["steps"], 4, True) for N, K in _sizes(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    size = 8 if case["precision"] == "fp64" else 4
    K = 2 * case["nx"] * case["ny"] - bool(case.get("odd"))
    steps = case.get("steps", 1)
    if case["kind"] == "solve":
        rough = {"mesh": _mesh(case["nx"], case["ny"], np.random.default_rng(0), False,
                               case["box"]), "N": case["N"], "eps": None}
        steps = math.ceil(case["T"] / _cfl_dt(rough))
    w = _work_of(case["N"], K, 5 * steps, size, bool(case.get("media")), case["kind"] == "rhs")
    if case["kind"] == "jobs":
        w = {k: v * case["jobs"] for k, v in w.items()}
    return w


# ------------------------------------------------------- the method in FP64
_A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238,
      -3550918686646 / 2091501179385, -1275806237668 / 842570457699)
_B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357,
      1720146321549 / 2090206949498, 3134564353537 / 4481467310338,
      2277821191437 / 14882151754819)
_BLEND = {1: 0.0, 2: 0.0, 3: 1.4152, 4: 0.1001, 5: 0.2751, 6: 0.98, 7: 1.0999}
_quad = np.longdouble


def _inverse(A):
    """Inverse in extended precision: Newton's iteration from the FP64 one."""
    X = np.linalg.inv(A.astype(np.float64)).astype(_quad)
    for _ in range(3):
        X = X @ (2 * np.eye(len(A), dtype=_quad) - A @ X)
    return X


def _bernstein(N, lam):
    """Bernstein polynomials of degree N and their derivatives along every
    barycentric coordinate: exponents, values [point, i], [coord][point, i]."""
    dims = len(lam)
    ex = [(i, N - i) for i in range(N + 1)] if dims == 2 else \
        [(i, j, N - i - j) for i in range(N + 1) for j in range(N + 1 - i)]
    lam = [np.asarray(v, _quad) for v in lam]
    V = np.zeros((len(lam[0]), len(ex)), _quad)
    D = [np.zeros_like(V) for _ in lam]
    for m, e in enumerate(ex):
        c = math.factorial(N) // math.prod(math.factorial(i) for i in e)
        V[:, m] = c * math.prod(v ** i for v, i in zip(lam, e))
        for d in range(dims):
            if e[d]:
                D[d][:, m] = c * e[d] * math.prod(v ** (i - (k == d))
                                                  for k, (v, i) in enumerate(zip(lam, e)))
    return ex, V, D


def _bernstein_mass(N, ex, volume):
    """Mass matrix of Bernstein polynomials on a simplex of that volume."""
    dim = len(ex[0]) - 1
    scale = _quad(volume) / (math.comb(2 * N, N) * math.comb(2 * N + dim, dim))
    return np.array([[math.prod(math.comb(i + j, i) for i, j in zip(a, b)) for b in ex]
                     for a in ex], _quad) * scale


class _Element:
    """Reference triangle (-1,-1), (1,-1), (-1,1): warp-and-blend nodes, Dr,
    Ds, LIFT, and each face's nodes counter-clockwise."""

    def __init__(self, N):
        lb = np.array([c / N for r in range(N + 1) for c in range(N + 1 - r)])
        lc = np.array([r / N for r in range(N + 1) for c in range(N + 1 - r)])
        la = 1 - lb - lc
        eq = np.linspace(-1, 1, N + 1)
        shift = np.polynomial.Polynomial.fit(eq, _edge_nodes(N) - eq, N, domain=[-1, 1])

        def warp(t):
            out = np.zeros_like(t)
            ok = np.abs(t) < 1 - 1e-10
            out[ok] = shift(t[ok]) / (1 - t[ok] ** 2)
            return out

        move = np.zeros((3, len(la)))  # of the three barycentric coordinates
        lam = np.stack([la, lb, lc])
        for i, j, k in ((0, 1, 2), (1, 2, 0), (2, 0, 1)):
            w = 2 * lam[i] * lam[j] * (1 + (_BLEND[N] * lam[k]) ** 2) * warp(lam[j] - lam[i])
            move[i] -= w
            move[j] += w
        lam = lam + move
        self.N, self.Np = N, len(la)
        self.r, self.s = 2 * lam[1] - 1, 2 * lam[2] - 1
        ex, V, D = _bernstein(N, lam)
        X = _inverse(V)
        self.X, self.ex = X, ex
        Dr, Ds = (D[1] - D[0]) / 2 @ X, (D[2] - D[0]) / 2 @ X
        at = {(round(c), round(r)): i for i, (c, r) in enumerate(zip(lb * N, lc * N))}
        self.faces = [[at[c, 0] for c in range(N + 1)], [at[N - r, r] for r in range(N + 1)],
                      [at[0, N - r] for r in range(N + 1)]]
        self.Minv = V @ _inverse(_bernstein_mass(N, ex, 2)) @ V.T
        g = _edge_nodes(N)
        ex1, V1, _ = _bernstein(N, ((1 - g) / 2, (1 + g) / 2))
        X1 = _inverse(V1)
        edge = X1.T @ _bernstein_mass(N, ex1, 2) @ X1
        E = np.zeros((self.Np, 3 * (N + 1)), _quad)
        for f, nodes in enumerate(self.faces):
            E[nodes, f * (N + 1):(f + 1) * (N + 1)] = edge
        self.Dr, self.Ds, self.LIFT = (torch.as_tensor(m.astype(np.float64)).cuda()
                                       for m in (Dr, Ds, self.Minv @ E))

    def at(self, r, s):
        """Nodal basis at one point."""
        _, v, _ = _bernstein(self.N, ([-(r + s) / 2], [(1 + r) / 2], [(1 + s) / 2]))
        return (v @ self.X)[0]


class _Reference:
    """Semi-discrete system of one problem, FP64 on the GPU."""

    def __init__(self, p):
        R = self.R = _Element(p["N"])
        x, y, E = p["mesh"]
        K, n = len(E), R.N + 1
        E = E.astype(np.int64)
        X, Y = x[E], y[E]
        xr, xs = (X[:, 1] - X[:, 0]) / 2, (X[:, 2] - X[:, 0]) / 2
        yr, ys = (Y[:, 1] - Y[:, 0]) / 2, (Y[:, 2] - Y[:, 0]) / 2
        J = xr * ys - xs * yr

        def col(v):
            return torch.as_tensor(v).cuda()[:, None]

        self.rx, self.ry, self.sx, self.sy = (col(v / J) for v in (ys, -xs, -yr, xr))
        L = np.stack([-(R.r + R.s) / 2, (1 + R.r) / 2, (1 + R.s) / 2])
        self.x, self.y = X @ L, Y @ L
        self.X, self.Y, self.J = X, Y, J
        tx, ty = np.roll(X, -1, 1) - X, np.roll(Y, -1, 1) - Y
        length = np.hypot(tx, ty)

        def per_node(v):
            return torch.as_tensor(v).cuda().repeat_interleave(n, 1)

        self.nx, self.ny = per_node(ty / length), per_node(-tx / length)
        self.scale = per_node(length / 2 / J[:, None])
        # a face's neighbour lists the shared nodes in reverse
        a, b = E, np.roll(E, -1, 1)
        key = (np.minimum(a, b) * len(x) + np.maximum(a, b)).ravel()
        order = np.argsort(key, kind="stable")
        same = np.nonzero(key[order][1:] == key[order][:-1])[0]
        other = np.arange(3 * K)
        other[order[same]], other[order[same + 1]] = order[same + 1], order[same]
        F = np.array(R.faces)
        self.own = torch.as_tensor((np.arange(K)[:, None] * R.Np + F.ravel()[None, :]).ravel()).cuda()
        wall = other == np.arange(3 * K)
        far = (other // 3 * R.Np)[:, None] + np.where(wall[:, None], F[other % 3],
                                                      F[other % 3][:, ::-1])
        self.far = torch.as_tensor(far.ravel()).cuda()
        self.wall = torch.as_tensor(wall).cuda().reshape(K, 3).repeat_interleave(n, 1)
        self.eps = None if p["eps"] is None else col(np.asarray(p["eps"], np.float64))
        z = np.ones(K) if p["eps"] is None else 1 / np.sqrt(p["eps"])
        self.zm, self.zp = col(z), per_node(z[other // 3].reshape(K, 3))
        self.load = None

    def source(self, sx, sy, f, t0, amplitude):
        X, Y = self.X, self.Y
        det = 4 * self.J
        l2 = ((sx - X[:, 0]) * (Y[:, 2] - Y[:, 0]) - (X[:, 2] - X[:, 0]) * (sy - Y[:, 0])) / det
        l3 = ((X[:, 1] - X[:, 0]) * (sy - Y[:, 0]) - (sx - X[:, 0]) * (Y[:, 1] - Y[:, 0])) / det
        k = int(np.nonzero((l2 >= -1e-12) & (l3 >= -1e-12) & (1 - l2 - l3 >= -1e-12))[0][0])
        w = self.R.Minv @ self.R.at(2 * l2[k] - 1, 2 * l3[k] - 1) / self.J[k]
        w = torch.as_tensor(w.astype(np.float64)).cuda()
        self.load = (k, w, f, t0, amplitude)

    def rhs(self, q, t=0.0):
        R = self.R
        hx, hy, ez = q
        n = self.own.numel()

        def jump(u):
            u = u.reshape(-1)
            return (u[self.own] - u[self.far]).reshape(-1, n // len(hx))

        jx, jy, je = jump(hx), jump(hy), jump(ez)
        inside = ez.reshape(-1)[self.own].reshape(je.shape)
        je = torch.where(self.wall, 2 * inside, je)
        jt = self.ny * jx - self.nx * jy
        both = self.zm + self.zp
        fz = (self.zp * jt - je) / both * self.scale
        g = -self.zm * fz

        def grad(u):
            ur, us = u @ R.Dr.T, u @ R.Ds.T
            return self.rx * ur + self.sx * us, self.ry * ur + self.sy * us

        ezx, ezy = grad(ez)
        out = torch.stack([(self.ny * g) @ R.LIFT.T - ezy, (-self.nx * g) @ R.LIFT.T + ezx,
                           fz @ R.LIFT.T + grad(hy)[0] - grad(hx)[1]])
        if self.eps is not None:
            out[2] /= self.eps
        if self.load is not None:
            k, w, f, t0, amplitude = self.load
            a = (math.pi * f * (t - t0)) ** 2
            out[2, k] += amplitude * (1 - 2 * a) * math.exp(-a) * w
        return out

    def steps(self, q, dt, count):
        q = q.clone()
        for m in range(count):
            res, c, clock = torch.zeros_like(q), 0.0, 0.0
            for a, b in zip(_A, _B):
                res = a * res + dt * self.rhs(q, (m + clock) * dt)
                c = a * c + 1.0
                clock += b * c
                q += b * res
        return q


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "server"):
        outs = []
        for p in _problems(case, seed):
            ref, dt, steps = _Reference(p), _cfl_dt(p), case["steps"]
            if kind == "batch":
                q = _fields(p, (ref.x, ref.y), torch.float32).double()
            else:
                q = torch.zeros((3,) + ref.x.shape, dtype=torch.float64, device="cuda")
                ref.source(*_ricker_of(p, dt, steps))
                dt *= (steps - 0.5) / steps
            outs.append(ref.steps(q, dt, steps))
        return outs
    p = _problem(case, seed)
    ref, dt, steps = _Reference(p), _cfl_dt(p), case.get("steps", 0)
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    q = _fields(p, (ref.x, ref.y), dtype)
    if kind == "rhs":
        return ref.rhs(q.double())
    if kind == "jobs":
        return [ref.steps((q / (j + 1)).double(), dt, steps) for j in range(case["jobs"])]
    if kind == "solve":
        steps = math.ceil(case["T"] / dt - 1e-12)
        dt = case["T"] / steps
    elif kind == "source":
        q = torch.zeros_like(q)
        ref.source(*_ricker_of(p, dt, steps))
        dt *= (steps - 0.5) / steps
    return ref.steps(q.double(), dt, steps)
