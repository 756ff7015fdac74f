"""The workloads this framework is timed on, each one pass through its public Python API.

`listed()` names them; `draw(rng)` gives further ones of the same ranges. `prepare` makes what a
program holds before the call (positions, right-hand sides, an uploaded mesh, options), `run` is
one pass, `exact` the same results from plain torch in 64 bits and `work` the bytes and operations
that a pass cannot do without.
"""
import math

import torch

from paper_2602_12105_gb300 import api, meshgen

DEV = "cuda"
LARGEST_GRID = 4096 * 2048


# ----------------------------------------------------------------------------------- the cases
def _smooth(name, mesh, nx, ny, t_rel, prec, tol, k=3, b="B", clamp=None, shuffle=False, upload=False):
    """Differentiable smoothing (api.smooth and backward). mesh "ico": nx is the level; "grid": nx x
    ny vertices. t_rel: the time step in units of the squared mean edge length. b "V": the
    positions themselves are smoothed. shuffle: vertices in random order, as in scanned or remeshed
    models. upload: the pass starts from the faces (a new topology in every pass)."""
    return {"name": name, "kind": "smooth", "mesh": mesh, "nx": nx, "ny": ny, "t_rel": t_rel, "prec": prec,
            "tol": tol, "k": k, "b": b, "clamp": clamp, "shuffle": shuffle, "upload": upload}


def listed():
    return [
        # The smallest mesh of the test-suite and the benchmark, to a tight tolerance: one small
        # model in an interactive loop, where launches and latency count.
        _smooth("ico3_fp64", "ico", 3, 0, 0.05, "fp64", 1e-12, b="V"),
        # An open patch with ragged sides and one scalar field on it (k = 1), a long time step;
        # gradients of the positions, the field and the step size.
        _smooth("grid97x61_fp64_k1", "grid", 97, 61, 30.0, "fp64", 1e-11, k=1),
        # The benchmark's default workload: a 1024 x 1024 height field in double precision.
        _smooth("grid1024_fp64", "grid", 1024, 1024, 1.0, "fp64", 1e-10),
        # The same in mixed precision.
        _smooth("grid1024_mixed", "grid", 1024, 1024, 1.0, "mixed", 1e-10),
        # The benchmark's largest mesh (8.4 million vertices), mixed precision.
        _smooth("grid4096x2048_mixed", "grid", 4096, 2048, 1.0, "mixed", 1e-10),
        # A large odd-sized height field with the FP32 face geometry option.
        _smooth("grid2047x1531_mixed32", "grid", 2047, 1531, 1.0, "mixed32", 1e-10),
        # A model in random vertex order whose topology is new in every pass (remeshing, or a
        # request of the server), with the cotangent clamp on.
        _smooth("shuffled601x419_new_mesh", "grid", 601, 419, 4.0, "mixed", 1e-10, b="V", clamp=0.0,
                shuffle=True, upload=True),
        # The differentiation batch of the benchmark: 256 icospheres of levels 2 to 6.
        {"name": "batch256_mixed", "kind": "batch", "count": 256, "lo": 2, "hi": 6, "prec": "mixed", "tol": 1e-10},
        # A smaller training batch in the default precision.
        {"name": "batch40_fp64", "kind": "batch", "count": 40, "lo": 2, "hi": 6, "prec": "fp64", "tol": 1e-10},
        # One step of the inverse-fairing optimisation on the benchmark's 163,842-vertex sphere.
        {"name": "fairing_ico7_fp64", "kind": "fairing", "level": 7, "t": 2e-3, "prec": "fp64", "tol": 1e-10},
        # Lowest eigenvectors of the same sphere by shift-invert iteration (k = 4).
        {"name": "eigs_ico7_k4", "kind": "eigs", "level": 7, "t": 0.5, "k": 4, "iters": 3, "tol": 1e-12},
        # Rounds of the geodesic-distance ADMM on the benchmark's flat 257 x 257 grid.
        {"name": "geodesic_grid257", "kind": "geodesic", "nx": 257, "ny": 257, "rounds": 4, "tol": 1e-13},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    p = rng.random()
    if p < 0.6:
        prec = rng.choice(["fp64", "mixed", "mixed32"])
        k = rng.choice([1, 2, 3, 3, 3, 4])
        if rng.random() < 0.3:
            level = rng.randint(2, 7)
            b = "V" if k == 3 and rng.random() < 0.5 else "B"
            return dict(_smooth("", "ico", level, 0, round(_log(rng, 0.05, 30.0), 4), prec, 1e-10, k=k, b=b))
        n = _log(rng, 600, 1.2e6 if prec == "fp64" else 0.9 * LARGEST_GRID)
        ratio = _log(rng, 0.5, 2.0)
        nx = max(5, round(math.sqrt(n * ratio)))
        ny = max(5, round(n / nx))
        t_rel = _log(rng, 0.3, 30.0 if n < 3e5 else 2.0)
        upload = n < 4e5 and rng.random() < 0.25
        shuffle = n < 2e6 and rng.random() < 0.3
        b = "V" if k == 3 and rng.random() < 0.4 else "B"
        clamp = 0.0 if rng.random() < 0.2 else None
        return dict(_smooth("", "grid", nx, ny, round(t_rel, 4), prec, 1e-10, k=k, b=b, clamp=clamp,
                            shuffle=shuffle, upload=upload))
    if p < 0.75:
        lo = rng.randint(2, 4)
        return {"kind": "batch", "count": round(_log(rng, 3, 160)), "lo": lo, "hi": rng.randint(lo, 6),
                "prec": rng.choice(["fp64", "mixed"]), "tol": 1e-10}
    if p < 0.85:
        return {"kind": "fairing", "level": rng.randint(3, 7), "t": round(_log(rng, 2e-4, 4e-3), 6),
                "prec": rng.choice(["fp64", "mixed"]), "tol": 1e-10}
    if p < 0.93:
        return {"kind": "eigs", "level": rng.randint(3, 6), "t": round(_log(rng, 0.1, 0.6), 4),
                "k": rng.randint(1, 4), "iters": rng.randint(1, 3), "tol": 1e-12}
    return {"kind": "geodesic", "nx": rng.randint(17, 200), "ny": rng.randint(17, 200),
            "rounds": rng.randint(2, 4), "tol": 1e-13}


# ----------------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _uniform(g, *shape):
    return 2.0 * torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64) - 1.0


def _ico(level, sigma, g):
    """A unit icosphere with radial noise: positions, faces, the clean positions, mean edge^2."""
    Vc, F = meshgen.icosphere(level)
    Vc, F = torch.from_numpy(Vc).to(DEV), torch.from_numpy(F).to(DEV)
    V = Vc * (1.0 + sigma * _normal(g, Vc.shape[0], 1))
    return V, F, Vc, 4.0 * math.pi / Vc.shape[0] * 1.1547


def _grid(nx, ny, g, amp=0.05):
    """A height-field grid with spacing h = 1 / (ny - 1); heights amp N(0, 1) under a 5 x 5 mean filter."""
    h = 1.0 / (ny - 1)
    i = torch.arange(nx, device=DEV, dtype=torch.int32)
    j = torch.arange(ny, device=DEV, dtype=torch.int32)
    z = _normal(g, 1, 1, ny, nx) * amp
    z = torch.nn.functional.avg_pool2d(torch.nn.functional.pad(z, (2, 2, 2, 2), mode="replicate"), 5, 1)[0, 0]
    x = (i.to(torch.float64) * h).expand(ny, nx)
    y = (j.to(torch.float64) * h)[:, None].expand(ny, nx)
    V = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1).contiguous()
    v00 = (j[:-1, None] * nx + i[None, :-1]).reshape(-1)
    F = torch.stack([v00, v00 + 1, v00 + nx + 1, v00, v00 + nx + 1, v00 + nx], 1).reshape(-1, 3).contiguous()
    return V, F, h * h


def _make_mesh(F, n, clamp):
    mesh = api.Mesh(F, n)
    if clamp is not None:
        mesh.set_cot_clamp(clamp)
    return mesh


def _smooth_inputs(case, seed):
    g = _gen(seed)
    if case["mesh"] == "ico":
        V, F, T, e2 = _ico(case["nx"], 0.01, g)
    else:
        V, F, e2 = _grid(case["nx"], case["ny"], g)
        T = None
    n = V.shape[0]
    if case["shuffle"]:
        perm = torch.randperm(n, generator=g, device=DEV)
        inv = torch.empty_like(perm)
        inv[perm] = torch.arange(n, device=DEV)
        V, F = V[perm].contiguous(), inv[F.to(torch.int64)].to(torch.int32)
        F = F[torch.randperm(F.shape[0], generator=g, device=DEV)].contiguous()
        T = None
    B = None if case["b"] == "V" else _uniform(g, n, case["k"])
    if T is None or case["b"] != "V":
        T = _uniform(g, n, case["k"]) if B is not None else V + 0.01 * _normal(g, n, 3)
    return V, F, B, T, case["t_rel"] * e2


def _batch_inputs(case, seed):
    g = _gen(seed)
    items, r = [], torch.rand(case["count"], 2, generator=g, device=DEV, dtype=torch.float64).cpu().numpy()
    for i in range(case["count"]):
        # levels in turn, so that each seed's batch has the same sizes in another order of t
        level = case["lo"] + i % (case["hi"] - case["lo"] + 1)
        V, F, T, _ = _ico(level, 0.02, g)
        items.append((V, F, T, float(math.exp(math.log(1e-4) + r[i, 0] * math.log(100.0)))))
    return items


def prepare(case, seed):
    opts = api.make_opts(rel_tol=case["tol"])
    s = {"case": case, "opts": opts}
    kind = case["kind"]
    if kind == "smooth":
        V, F, B, T, t = _smooth_inputs(case, seed)
        s.update(V=V.requires_grad_(True), F=F, B=B.requires_grad_(True) if B is not None else None, T=T,
                 t=torch.tensor(t, dtype=torch.float64, requires_grad=True) if case["k"] == 1 else t)
        if not case["upload"]:
            s["mesh"] = _make_mesh(F, V.shape[0], case["clamp"])
    elif kind == "batch":
        items = _batch_inputs(case, seed)
        s["Vs"] = [V.requires_grad_(True) for V, _, _, _ in items]
        s["Ts"] = [T for _, _, T, _ in items]
        s["ts"] = [t for _, _, _, t in items]
        s["batch"] = api.Batch([api.Mesh(F, V.shape[0]) for V, F, _, _ in items])
    elif kind == "fairing":
        T, F, _, _ = _ico(case["level"], 0.02, _gen(seed))
        s["V0"], s["V"] = T.clone(), T.clone()
        s["fair"] = api.InverseFairing(api.Mesh(F, T.shape[0]), T, case["t"], 1.0, precision=case["prec"], opts=opts)
    elif kind == "eigs":
        g = _gen(seed)
        V, F, _, _ = _ico(case["level"], 0.002, g)
        s.update(V=V, U0=_uniform(g, V.shape[0], case["k"]), mesh=api.Mesh(F, V.shape[0]))
    else:
        g = _gen(seed)
        V, F, _ = _grid(case["nx"], case["ny"], g, amp=0.0)
        V[:, :2] += 0.1 / (case["ny"] - 1) * _uniform(g, V.shape[0], 2)
        s.update(V=V, mesh=api.Mesh(F, V.shape[0]))
    return s


# ----------------------------------------------------------------------------------- one pass
def run(s):
    case, opts = s["case"], s["opts"]
    kind = case["kind"]
    if kind == "smooth":
        V, B, t = s["V"], s["B"], s["t"]
        mesh = s["mesh"] if "mesh" in s else _make_mesh(s["F"], V.shape[0], case["clamp"])
        U = api.smooth(mesh, V, B, t, precision=case["prec"], opts=opts)
        wrt = [V] + ([B] if B is not None else []) + ([t] if isinstance(t, torch.Tensor) else [])
        grads = torch.autograd.grad(U, wrt, U.detach() - s["T"])
        if "mesh" not in s:
            mesh.close()
        return (U.detach(),) + tuple(grads)
    if kind == "batch":
        Us = api.smooth_batch(s["batch"], s["Vs"], None, s["ts"], precision=case["prec"], opts=opts)
        gs = torch.autograd.grad(Us, s["Vs"], [U.detach() - T for U, T in zip(Us, s["Ts"])])
        return torch.cat([U.detach() for U in Us]), torch.cat(gs)
    if kind == "fairing":
        s["V"].copy_(s["V0"])
        loss = s["fair"].step(s["V"])
        return s["V"], loss
    if kind == "eigs":
        s["mesh"].assemble(s["V"], case["t"])
        return s["mesh"].eigs(s["U0"], case["iters"], opts=opts)
    u, y, z, _ = s["mesh"].rgd_admm(s["V"], [0], 10.0, 0.0, 1.0, case["rounds"], opts=opts)
    return u, y, z


# ----------------------------------------------------------------------------------- what a pass needs
def _size(case):
    """Vertices, faces and columns of the case."""
    if case["kind"] == "batch":
        lv = [case["lo"] + i % (case["hi"] - case["lo"] + 1) for i in range(case["count"])]
        return sum(10 * 4 ** v + 2 for v in lv), sum(20 * 4 ** v for v in lv), 3
    if case["kind"] in ("fairing", "eigs") or case.get("mesh") == "ico":
        v = case["nx"] if case["kind"] == "smooth" else case["level"]
        return 10 * 4 ** v + 2, 20 * 4 ** v, case.get("k", 3)
    nx, ny = case["nx"], case["ny"]
    return nx * ny, 2 * (nx - 1) * (ny - 1), case.get("k", 1)


def work(case):
    """Each input read and each output written once; per solve the operations of a conjugate-gradient
    run of the length that the operator's condition number and the tolerance ask for (two
    operations for each of the 7 entries of a row and 15 for the vectors, per column and step),
    and about 350 operations per face for the operator and the gradient."""
    n, m, k = _size(case)
    kind = case["kind"]
    if kind == "geodesic":
        steps, solves = 2.0 * max(case["nx"], case["ny"]), case["rounds"]
        io = 24 * n + 12 * m + 8 * n + 48 * m
    else:
        if kind == "smooth":
            t_rel = case["t_rel"]
        elif kind == "batch":
            t_rel = 1e-3 * n / case["count"] / 14.5
        else:
            t_rel = case["t"] * n / 14.5
        steps = 0.5 * math.sqrt(1.0 + 8.0 * t_rel) * math.log(2.0 / case["tol"])
        solves = {"smooth": 2, "batch": 2, "fairing": 3}.get(kind) or case["iters"]
        fields = {"smooth": 2 + 2 * (case.get("b") == "B"), "batch": 2, "fairing": 1, "eigs": 2}[kind]
        io = 24 * n * (2 if kind != "eigs" else 1) + 12 * m + 8 * n * k * fields
    return {"bytes": io, "flops": solves * steps * n * k * (14 + 15) + 350.0 * m}


# ----------------------------------------------------------------------------------- 64-bit results
def _weights(V, F, t, clamp=None):
    """Per face: t cot / 2 of the three corners and area / 3."""
    p = V[F]
    d = [p[:, 2] - p[:, 1], p[:, 0] - p[:, 2], p[:, 1] - p[:, 0]]
    s = torch.linalg.vector_norm(torch.linalg.cross(d[1], d[2], dim=1), dim=1)
    w = torch.stack([-(d[(c + 1) % 3] * d[(c + 2) % 3]).sum(1) / s for c in range(3)], 1)
    if clamp is not None:
        w = w.clamp(min=clamp)
    return 0.5 * t * w, s / 6.0


def _csr(F, w, a3, n):
    """M + t L as a sparse matrix, and the mass."""
    M = torch.zeros(n, dtype=torch.float64, device=DEV)
    rows, cols, vals = [], [], []
    for c in range(3):
        a, b = F[:, (c + 1) % 3], F[:, (c + 2) % 3]
        M.index_add_(0, F[:, c], a3)
        rows += [a, b, a, b]
        cols += [b, a, a, b]
        vals += [-w[:, c], -w[:, c], w[:, c], w[:, c]]
    i = torch.arange(n, device=DEV)
    A = torch.sparse_coo_tensor(torch.stack([torch.cat(rows + [i]), torch.cat(cols + [i])]),
                                torch.cat(vals + [M]), (n, n)).coalesce()
    ij = A.indices()
    D = torch.zeros(n, dtype=torch.float64, device=DEV)
    on = ij[0] == ij[1]
    D[ij[0][on]] = A.values()[on]
    return A.to_sparse_csr(), M, D


def _solve(A, D, B, X=None):
    """A X = B by Jacobi-preconditioned conjugate gradients, restarted until the residual is rounding."""
    X = torch.zeros_like(B) if X is None else X
    b2 = (B * B).sum(0).clamp_min(1e-300)
    for _ in range(3):
        R = B - A @ X
        if float(((R * R).sum(0) / b2).max()) < 1e-30:
            break
        Z = R / D[:, None]
        P, rz = Z.clone(), (R * Z).sum(0)
        for it in range(20000):
            Q = A @ P
            al = torch.nan_to_num(rz / (P * Q).sum(0))
            X = X + al * P
            R = R - al * Q
            Z = R / D[:, None]
            rz, old = (R * Z).sum(0), rz
            P = Z + torch.nan_to_num(rz / old) * P
            if it % 10 == 9 and float(((R * R).sum(0) / b2).max()) < 1e-32:
                break
    return X


def _gradient(V, F, B, U, Lam, t, clamp, extra=None):
    """d/d(V, t, B) of <Lam, M B - (M + t L) U> (+ extra(mass)); B None: the positions."""
    V = V.detach().clone().requires_grad_(True)
    Bv = V if B is None else B.detach().clone().requires_grad_(True)
    tt = t.detach().clone().requires_grad_(True) if isinstance(t, torch.Tensor) else \
        torch.tensor(t, dtype=torch.float64, device=DEV, requires_grad=True)
    total = [torch.zeros_like(V), torch.zeros_like(Bv), torch.zeros_like(tt)]
    step = 4_000_000
    for f0 in range(0, F.shape[0], step):
        f = F[f0:f0 + step]
        w, a3 = _weights(V, f, tt, clamp)
        e = (a3[:, None] * (Lam * (Bv - U)).sum(1)[f]).sum()
        if extra is not None:
            e = e + (a3[:, None] * extra[f]).sum()
        for c in range(3):
            a, b = f[:, (c + 1) % 3], f[:, (c + 2) % 3]
            e = e - (w[:, c] * ((Lam[a] - Lam[b]) * (U[a] - U[b])).sum(1)).sum()
        for x, y in zip(total, torch.autograd.grad(e, (V, Bv, tt), allow_unused=True)):
            if y is not None:
                x += y
    return total


def exact(case, seed):
    kind = case["kind"]
    if kind == "smooth":
        V, F, B, T, t = _smooth_inputs(case, seed)
        F, n = F.to(torch.int64), V.shape[0]
        A, M, D = _csr(F, *_weights(V, F, t, case["clamp"]), n)
        U = _solve(A, D, M[:, None] * (V if B is None else B))
        Lam = _solve(A, D, U - T)
        gV, gB, gt = _gradient(V, F, B, U, Lam, t, case["clamp"])
        return (U, gV) + ((gB,) if B is not None else ()) + ((gt,) if case["k"] == 1 else ())
    if kind == "batch":
        items = _batch_inputs(case, seed)
        V, T = torch.cat([i[0] for i in items]), torch.cat([i[2] for i in items])
        off, Fs, ts = 0, [], []
        for v, f, _, t in items:
            Fs.append(f.to(torch.int64) + off)
            ts.append(torch.full((f.shape[0],), t, dtype=torch.float64, device=DEV))
            off += v.shape[0]
        F, t = torch.cat(Fs), torch.cat(ts)
        A, M, D = _csr(F, *_weights(V, F, t[:, None]), off)
        U = _solve(A, D, M[:, None] * V)
        Lam = _solve(A, D, U - T)
        gV = torch.zeros_like(V)
        for v, f, tm in zip(range(len(items)), Fs, [i[3] for i in items]):
            a, b = int(f.min()), int(f.max()) + 1
            gV[a:b] = _gradient(V[a:b], f - a, None, U[a:b], Lam[a:b], tm, None)[0]
        return U, gV
    if kind == "fairing":
        T, F, _, _ = _ico(case["level"], 0.02, _gen(seed))
        F = F.to(torch.int64)
        A, M, D = _csr(F, *_weights(T, F, case["t"]), T.shape[0])
        U = _solve(A, D, M[:, None] * T)
        e = 0.5 * ((U - T) ** 2).sum(1)
        Lam = _solve(A, D, M[:, None] * (U - T))
        g = _gradient(T, F, None, U, Lam, case["t"], None, extra=e)[0]
        return T - _solve(A, D, g), (M * e).sum()
    if kind == "eigs":
        g = _gen(seed)
        V, F, _, _ = _ico(case["level"], 0.002, g)
        U = _uniform(g, V.shape[0], case["k"])
        F = F.to(torch.int64)
        A, M, D = _csr(F, *_weights(V, F, case["t"]), V.shape[0])
        for _ in range(case["iters"]):
            Y = _solve(A, D, M[:, None] * U)
            R = torch.linalg.cholesky(Y.T @ (M[:, None] * Y)).T
            U = torch.linalg.solve_triangular(R.T, Y.T, upper=False).T
        top = U.abs() >= (1.0 - 1e-6) * U.abs().max(0).values
        first = top.to(torch.int8).argmax(0)
        U = U * torch.sign(U[first, torch.arange(U.shape[1], device=DEV)])
        lam = ((U * (A @ U)).sum(0) - (M[:, None] * U * U).sum(0)) / case["t"]
        return U, lam
    return _exact_geodesic(case, seed)


def _exact_geodesic(case, seed):
    g = _gen(seed)
    V, F, _ = _grid(case["nx"], case["ny"], g, amp=0.0)
    V[:, :2] += 0.1 / (case["ny"] - 1) * _uniform(g, V.shape[0], 2)
    F, n, rho = F.to(torch.int64), V.shape[0], 10.0
    w, a3 = _weights(V, F, 1.0)
    keep = torch.ones(n, dtype=torch.float64, device=DEV)
    keep[0] = 0.0
    _, M, _ = _csr(F, w, a3, n)
    A, _, D = _csr(F, w, torch.zeros_like(a3), n)
    coo = A.to_sparse_coo().coalesce()
    i, j = coo.indices()
    vals = torch.where((i == 0) | (j == 0), (i == j).to(torch.float64), coo.values())
    A = torch.sparse_coo_tensor(coo.indices(), vals, (n, n)).coalesce().to_sparse_csr()
    D = D * keep + (1.0 - keep)
    p = V[F]
    N = torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0], dim=1)
    N2 = (N * N).sum(1, keepdim=True)
    grad = [torch.linalg.cross(N, p[:, (c + 2) % 3] - p[:, (c + 1) % 3], dim=1) / N2 for c in range(3)]
    area = 0.5 * torch.sqrt(N2)
    y, z = torch.zeros_like(N), torch.zeros_like(N)
    u = torch.zeros(n, 1, dtype=torch.float64, device=DEV)
    for _ in range(case["rounds"]):
        b = M.clone()
        for c in range(3):
            b.index_add_(0, F[:, c], -(area * grad[c] * (y - rho * z)).sum(1))
        u = _solve(A, D, (b * keep / rho)[:, None], u)
        gu = sum(u[F[:, c]] * grad[c] for c in range(3))
        z = y / rho + gu
        z = z / torch.linalg.vector_norm(z, dim=1, keepdim=True).clamp_min(1.0)
        y = y + rho * (gu - z)
    return u[:, 0], y, z
