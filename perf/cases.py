"""Performance cases: the work that users of this library have it do, through its
public entry points.

Four kinds, over the ranges of the repository's own configurations, tests and
benchmark:

  residual  F(u) of a context (bfs_residual), double-float and FP64 pair sums
  solve     Newton-Krylov solves: the uniform stream or the guess network as the
            start, a new topography on a factored context, a new (mesh, F) whose
            preconditioner is factored first, and the plain FP64 default options
  factor    the default (FP64) preconditioner factored and applied once
  batch     many uneven meshes solved in lockstep
  train     loss and gradient of the guess network on one training batch

Every solve stops at |F|_inf <= 1e-10, so that its answer does not depend on
the path Newton took to it.
"""
import math

import numpy as np
import torch

from paper_1709_08803_gb300 import bfs, surrogate
from paper_1709_08803_gb300 import workloads as W

TOL = 1e-10
LAYERS = ((16, 32, 1), (32, 32, 3), (32, 32, 9), (32, 16, 27))  # cin, cout, dilation


def listed():
    return [
        # the smallest residual call: the half-domain test mesh, where launches and latency count
        {"name": "residual df64 31x11 half", "kind": "residual", "N": 31, "M": 11, "half": 1, "dx": 0.4, "precision": "df64"},
        # the FP64-accurate Newton residual of the benchmark mesh
        {"name": "residual df64 181x61", "kind": "residual", "N": 181, "M": 61, "half": 0, "dx": 0.3, "precision": "df64"},
        # the paper's own mesh (Sec. 5): the largest residual a user evaluates
        {"name": "residual df64 281x281", "kind": "residual", "N": 281, "M": 281, "half": 0, "dx": 24.0 / 280.0, "precision": "df64"},
        # the default arithmetic of bfs_residual, on the benchmark mesh
        {"name": "residual fp64 181x61", "kind": "residual", "N": 181, "M": 61, "half": 0, "dx": 0.3, "precision": "fp64"},
        # a solve with nothing but defaults (FP64 throughout) on the half-domain test mesh
        {"name": "solve default 31x11 half", "kind": "solve", "start": "flat", "form": "default", "N": 31, "M": 11, "half": 1, "dx": 0.4, "F": 0.7},
        # the benchmark's headline: guess network, then the mixed-precision solve, subcritical
        {"name": "solve learned 181x61", "kind": "solve", "start": "learned", "form": "mixed", "N": 181, "M": 61, "half": 0, "dx": 0.3, "F": 0.7},
        # the benchmark's supercritical configuration: long Krylov cycles
        {"name": "solve mixed 181x61 F1.5", "kind": "solve", "start": "flat", "form": "mixed", "N": 181, "M": 61, "half": 0, "dx": 0.3, "F": 1.5},
        # the first solve of a new (mesh, F): factorisation and solve, odd sizes
        {"name": "first solve 151x53", "kind": "solve", "start": "factor", "form": "mixed", "N": 151, "M": 53, "half": 0, "dx": 0.3, "F": 0.6},
        # a continuation step (new topography, factored context) on the widest batched-sweep mesh
        {"name": "continuation 241x81", "kind": "solve", "start": "topography", "form": "mixed", "N": 241, "M": 81, "half": 0, "dx": 0.3, "F": 0.6},
        # the preconditioner with default options: FP64 factors, FP64 sweeps
        {"name": "factor default 181x61", "kind": "factor", "N": 181, "M": 61, "half": 0, "dx": 0.3, "F": 0.7},
        # a batched sweep over uneven meshes
        {"name": "batch solve 12", "kind": "batch", "B": 12, "Nlo": 61, "Nhi": 161},
        # one training batch of the guess network
        {"name": "train 16 at 181x61", "kind": "train", "B": 16, "N": 181, "M": 61},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("residual", "residual", "residual", "solve", "solve", "factor", "batch", "train"))
    if kind == "residual":
        if rng.random() < 0.6:
            N, M = _log_int(rng, 21, 281), _log_int(rng, 7, 240)
            return {"kind": kind, "N": N, "M": M, "half": 0, "dx": rng.choice((24.0 / 280.0, 0.2, 0.3, 0.4)), "precision": "df64"}
        N, M = _log_int(rng, 21, 181), _log_int(rng, 7, 61)
        half = rng.choice((0, 1)) if M <= 31 else 0
        return {"kind": kind, "N": N, "M": M, "half": half, "dx": rng.choice((0.2, 0.3, 0.4)), "precision": rng.choice(("df64", "fp64"))}
    if kind == "solve":
        N = _log_int(rng, 61, 201)
        F = rng.uniform(0.5, 0.68) if rng.random() < 0.75 else rng.uniform(1.45, 1.6)
        return {"kind": kind, "start": rng.choice(("flat", "factor", "topography")), "form": "mixed", "N": N,
                "M": (N - 1) // 3 + rng.choice((0, 1, 2)), "half": 0, "dx": 0.3, "F": F}
    if kind == "factor":
        N = _log_int(rng, 31, 181)
        return {"kind": kind, "N": N, "M": (N - 1) // 3 + rng.choice((0, 1, 2)), "half": 0, "dx": 0.3, "F": rng.uniform(0.5, 1.5)}
    if kind == "batch":
        return {"kind": kind, "B": rng.randint(3, 12), "Nlo": rng.choice((31, 45, 61)), "Nhi": rng.choice((91, 121, 161))}
    return {"kind": kind, "B": rng.randint(1, 16), "N": _log_int(rng, 61, 181), "M": _log_int(rng, 21, 61)}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _mesh(case):
    if case["half"]:
        return W.Mesh(N=case["N"], M=case["M"], x1=-0.5 * (case["N"] - 1) * case["dx"], y1=0.0, dx=case["dx"], dy=case["dx"], half=1)
    return W.mesh_box(case["N"], case["M"], case["dx"], case["dx"])


def _bumps(rng, half=0, scale=1.0):
    """One Gaussian near the benchmark's (height 0.2, delta = 1/sqrt(2), at the origin)."""
    return [(scale * float(rng.uniform(0.12, 0.2)), float(rng.uniform(0.6, 0.75)), float(rng.uniform(-0.5, 0.5)),
             0.0 if half else float(rng.uniform(-0.5, 0.5)))]


def _options(case):
    if case["form"] == "default":
        return bfs.default_options(tol=TOL)
    return bfs.default_options(tol=TOL, krylov_precision=bfs.BFS_FP32C, outer_precision=bfs.BFS_DF64, eta=1e-2,
                               refine_below=1e-5, precond_precision=bfs.BFS_FP32C, forcing=1, max_krylov=400)


PRECISION = {"fp64": bfs.BFS_FP64, "df64": bfs.BFS_DF64}


def _residual_inputs(case, seed):
    mesh, rng = _mesh(case), np.random.default_rng(seed)
    return mesh, W.gaussian_bumps(mesh, _bumps(rng, case["half"])), 0.7, W.smooth_guess(mesh, seed)


def _solve_inputs(case, seed):
    mesh, rng = _mesh(case), np.random.default_rng(seed)
    bumps = _bumps(rng, case["half"])
    return mesh, W.gaussian_bumps(mesh, bumps), W.gaussian_bumps(mesh, [(0.8 * b[0], *b[1:]) for b in bumps])


def _batch_inputs(case, seed):
    rng = np.random.default_rng(seed)
    meshes, topos, Fs = [], [], []
    for i in range(case["B"]):
        N = case["Nlo"] + (case["Nhi"] - case["Nlo"]) * i // max(1, case["B"] - 1)
        mesh = W.mesh_box(N, (N - 1) // 3 + 1, 0.3, 0.3)
        meshes.append(mesh)
        topos.append(W.gaussian_bumps(mesh, _bumps(rng, scale=0.6)))
        Fs.append(float(rng.uniform(0.5, 0.62)))
    return meshes, topos, Fs


def _factor_inputs(case, seed):
    mesh, rng = _mesh(case), np.random.default_rng(seed)
    return mesh, W.gaussian_bumps(mesh, _bumps(rng, case["half"])), case["F"], rng.standard_normal(mesh.n_unknowns)


def _train_inputs(case, seed):
    mesh, rng = W.mesh_box(case["N"], case["M"], 0.3, 0.3), np.random.default_rng(seed)
    x = np.stack([surrogate.features(mesh, W.gaussian_bumps(mesh, _bumps(rng)), float(rng.uniform(0.5, 1.4)))
                  for _ in range(case["B"])])
    X, Y = np.meshgrid(mesh.x(), mesh.y())
    t = np.empty((case["B"], mesh.M, mesh.N, 3), dtype=np.float32)
    for b in range(case["B"]):
        for f in range(3):
            k1, k2, ph = rng.uniform(0.8, 2.5), rng.uniform(0.2, 1.2), rng.uniform(0, 2 * math.pi)
            t[b, :, :, f] = rng.uniform(0.5, 1.5) * np.cos(k1 * X + ph) * np.cos(k2 * Y)
    return x, t, surrogate.init_params(seed % 100000)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "residual":
        mesh, topo, F, u = _residual_inputs(case, seed)
        ctx = bfs.Context(mesh, topo, F)
        return {"kind": kind, "ctx": ctx, "u": torch.tensor(u, device="cuda"), "precision": PRECISION[case["precision"]]}
    if kind == "solve":
        mesh, topo, before = _solve_inputs(case, seed)
        start = case["start"]
        ctx = bfs.Context(mesh, before if start == "topography" else topo, case["F"], _options(case))
        s = {"kind": kind, "start": start, "ctx": ctx, "topo": topo}
        if start != "factor":
            ctx.precond_factor()
        if start == "learned":
            params, scale = surrogate.load()
            s["net"] = surrogate.CNO(mesh.M, mesh.N, 1)
            s["net"].set_params(params, scale)
            s["x"] = torch.tensor(surrogate.features(mesh, topo, case["F"])[None], device="cuda")
        if start == "topography":  # the solution of the continuation's previous stage
            s["u0"] = ctx.flat_guess()
            ctx.solve(s["u0"])
        return s
    if kind == "factor":
        mesh, topo, F, r = _factor_inputs(case, seed)
        return {"kind": kind, "ctx": bfs.Context(mesh, topo, F), "r": torch.tensor(r, device="cuda")}
    if kind == "batch":
        meshes, topos, Fs = _batch_inputs(case, seed)
        b = bfs.Batch(meshes, topos, Fs, _options({"form": "mixed"}))
        for i in range(b.B):  # each instance's preconditioner, as a sweep over many bottoms keeps it
            b._check(bfs.lib().bfs_precond_factor(bfs.lib().bfs_batch_instance(b._b, i), -1, bfs._stream(None)))
        return {"kind": kind, "batch": b}
    x, t, p = _train_inputs(case, seed)
    net = surrogate.CNO(case["M"], case["N"], case["B"])
    net.set_params(p)
    return {"kind": kind, "net": net, "x": torch.tensor(x, device="cuda"), "t": torch.tensor(t, device="cuda")}


def run(state):
    kind = state["kind"]
    if kind == "residual":
        return state["ctx"].residual(state["u"], precision=state["precision"])
    if kind == "solve":
        ctx, start = state["ctx"], state["start"]
        if start == "learned":
            u = torch.empty(ctx.n, dtype=torch.float64, device="cuda")
            st = state["net"].solve(ctx, state["x"], u)
            if st["status"] != bfs.BFS_OK:
                raise RuntimeError(f"no convergence: {st}")
            return u
        if start == "topography":
            ctx.set_topography(state["topo"])
            u = state["u0"].clone()
        else:
            if start == "factor":
                ctx.precond_factor()
            u = ctx.flat_guess()
        ctx.solve(u)
        return u
    if kind == "factor":
        state["ctx"].precond_factor()
        return state["ctx"].precond_apply(state["r"])
    if kind == "batch":
        us = state["batch"].flat_guesses()
        state["batch"].solve(us, raise_on_error=True)
        return us
    g, loss = state["net"].gradient(state["x"], state["t"])
    return {"gradient": g, "loss": loss}


# ---------------------------------------------------------------------------
# Work one pass cannot do without
# ---------------------------------------------------------------------------
PAIR_FLOPS = 60  # floating-point operations of one (half point, node) pair, both sheets of each


def _pairs(mesh):
    return float(mesh.n_targets) * mesh.n_sources


def _band(mesh, itemsize):
    """Bytes of the block-banded factors and the operations of their block LU."""
    h, nb = max(1, round(mesh.M / 20.0)), 3.0 * (mesh.N + 1)
    return mesh.M * (2 * h + 1) * nb * nb * itemsize, mesh.M * nb ** 3 * 2.0 * (1 + 2 * h + h * h)


def work(case):
    kind = case["kind"]
    if kind == "train":
        P = case["B"] * case["N"] * case["M"]
        macs = sum(9 * a * b for a, b, _ in LAYERS)
        weights = macs + sum(b for _, b, _ in LAYERS)
        return {"bytes": P * 7 * 4 + weights * 4 * 2, "flops": 6.0 * P * macs}
    if kind == "batch":
        meshes = _batch_inputs(case, 0)[0]
        return {"bytes": sum(50 * _band(m, 4)[0] for m in meshes), "flops": sum(50 * _pairs(m) * PAIR_FLOPS for m in meshes)}
    mesh = _mesh(case)
    if kind == "residual":
        return {"bytes": 8 * (2 * mesh.n_unknowns + 3 * mesh.N * mesh.M), "flops": _pairs(mesh) * PAIR_FLOPS}
    fbytes, fflops = _band(mesh, 8)
    if kind == "factor":
        return {"bytes": 2 * fbytes + 16 * mesh.n_unknowns, "flops": fflops}
    its = 60 if case["F"] < 1 else 200  # Krylov steps, each a residual and a sweep over the factors
    return {"bytes": its * fbytes / 2, "flops": its * _pairs(mesh) * PAIR_FLOPS + (fflops if case["start"] == "factor" else 0.0)}


# ---------------------------------------------------------------------------
# 64-bit references in plain torch
# ---------------------------------------------------------------------------
def _dev(a):
    return torch.as_tensor(a, dtype=torch.float64, device="cuda")


def _ydiff(q, mesh):
    d = torch.empty_like(q)
    d[1:-1] = (q[2:] - q[:-2]) / (2 * mesh.dy)
    d[0] = 0.0 if mesh.half else (-3 * q[0] + 4 * q[1] - q[2]) / (2 * mesh.dy)
    d[-1] = (3 * q[-1] - 4 * q[-2] + q[-3]) / (2 * mesh.dy)
    return d


def _rect(A, B, C, mesh, xs, ys):
    """Closed form of the integral of (A s^2 + B s t + C t^2)^(-1/2) over the mesh rectangle."""
    xhi, yhi = mesh.x1 + (mesh.N - 1) * mesh.dx, mesh.y1 + (mesh.M - 1) * mesh.dy
    ylo = -yhi if mesh.half else mesh.y1
    D = 4 * A * C - B * B

    def term(a, c, s, t):  # t / sqrt(a) ln(2 a s + B t + 2 sqrt(a Q)), 0 at t = 0
        r = 2 * torch.sqrt(a * (a * s * s + B * s * t + c * t * t))
        lin = 2 * a * s + B * t
        v = t / torch.sqrt(a) * torch.log(torch.where(lin >= 0, lin + r, D * t * t / (r - lin)))
        return torch.where(t == 0, torch.zeros_like(v), v)

    out = 0.0
    for sgn, ex, ey in ((1, xhi, yhi), (-1, mesh.x1, yhi), (-1, xhi, ylo), (1, mesh.x1, ylo)):
        s, t = ex - xs, ey - ys
        out = out + sgn * (term(A, C, s, t) + term(C, A, t, s))
    return out


def _residual_exact(mesh, topo, F, u, n_rad=0.05, sigma=-1.0):
    N, M, dx, dy = mesh.N, mesh.M, mesh.dx, mesh.dy
    U = u.view(3, M, N + 1)
    q0, qx = U[:, :, :1], U[:, :, 1:]
    inc = torch.cumsum(0.5 * dx * (qx[:, :, 1:] + qx[:, :, :-1]), dim=2)
    nodal = torch.cat([q0, q0 + inc], dim=2)
    z, ph, ps = nodal
    zx, phx = qx[0], qx[1]
    zy, phy = _ydiff(z, mesh), _ydiff(ph, mesh)
    x = mesh.x1 + dx * torch.arange(N, dtype=torch.float64, device="cuda")
    y = mesh.y1 + dy * torch.arange(M, dtype=torch.float64, device="cuda")
    X, Y = x.expand(M, N), y.view(M, 1).expand(M, N)
    be, bx, by = (_dev(a).view(M, N) for a in (topo.beta, topo.beta_x, topo.beta_y))
    f, g = ph - X, ps - X
    cx = torch.ones(N, dtype=torch.float64, device="cuda")
    cx[0] = cx[-1] = 0.5
    cy = torch.ones(M, dtype=torch.float64, device="cuda")
    cy[-1] = 0.5
    if not mesh.half:
        cy[0] = 0.5
    w = dx * dy * cx * cy.view(M, 1)

    def sources(a, odd=False):  # nodes, then in the half domain their images at -y
        a = a.contiguous()
        return torch.cat([a.reshape(-1), (-a[1:] if odd else a[1:]).reshape(-1)]) if mesh.half else a.reshape(-1)

    S = {k: sources(a, k in ("y", "zy", "by")) for k, a in
         dict(x=X, y=Y, z=z, b=be, zx=zx, zy=zy, bx=bx, by=by, f=f, g=g, w=w).items()}
    half = lambda a: 0.5 * (a[:, 1:] + a[:, :-1])  # noqa: E731
    T = {k: half(a).reshape(-1, 1) for k, a in
         dict(x=X, y=Y, z=z, b=be, zx=zx, zy=zy, phx=phx, phy=phy, f=f, g=g, bx=bx, by=by).items()}
    Nt, Ns = (N - 1) * M, S["x"].numel()
    top = torch.empty(Nt, dtype=torch.float64, device="cuda")
    bot, s2t, cb = torch.empty_like(top), torch.empty_like(top), torch.empty_like(top)
    step = max(1, (1 << 26) // Ns)
    wf, wg, wzx, wbx = S["w"] * S["f"], S["w"] * S["g"], S["w"] * S["zx"], sigma * S["w"] * S["bx"]
    for a in range(0, Nt, step):
        t = {k: v[a:a + step] for k, v in T.items()}
        sx, sy = S["x"] - t["x"], S["y"] - t["y"]
        rho2 = sx * sx + sy * sy
        gt, gb = sx * S["zx"] + sy * S["zy"], sx * S["bx"] + sy * S["by"]
        d = S["z"] - t["z"]
        ri = torch.rsqrt(rho2 + d * d)
        acc = ((wf - t["f"] * S["w"]) * (d - gt) * ri ** 3 + wzx * ri).sum(1)
        d = S["b"] - t["z"]
        ri = torch.rsqrt(rho2 + d * d)
        top[a:a + step] = acc + (wbx * ri - wg * (d - gb) * ri ** 3).sum(1)
        d = S["z"] - t["b"]
        ri = torch.rsqrt(rho2 + d * d)
        acc = (wf * (d - gt) * ri ** 3 + wzx * ri).sum(1)
        d = S["b"] - t["b"]
        ri = torch.rsqrt(rho2 + d * d)
        bot[a:a + step] = acc - ((wg - t["g"] * S["w"]) * (d - gb) * ri ** 3).sum(1)
        m = sx * t["zx"] + sy * t["zy"]
        s2t[a:a + step] = (S["w"] * torch.rsqrt(rho2 + m * m)).sum(1)
        m = sx * t["bx"] + sy * t["by"]
        cb[a:a + step] = (wbx * ri - sigma * t["bx"] * S["w"] * torch.rsqrt(rho2 + m * m)).sum(1)
    t = {k: v.reshape(-1) for k, v in T.items()}
    rect = lambda p, q: _rect(1 + p * p, 2 * p * q, 1 + q * q, mesh, t["x"], t["y"])  # noqa: E731
    F2 = top - t["zx"] * s2t + t["zx"] * rect(t["zx"], t["zy"]) - 2 * math.pi * t["f"]
    F7 = bot + cb + sigma * t["bx"] * rect(t["bx"], t["by"]) - 2 * math.pi * t["g"]
    zx_, zy_, px, py = t["zx"], t["zy"], t["phx"], t["phy"]
    num = (1 + zx_ ** 2) * py ** 2 + (1 + zy_ ** 2) * px ** 2 - 2 * zx_ * zy_ * px * py
    F1 = 0.5 * num / (1 + zx_ ** 2 + zy_ ** 2) + t["z"] / F ** 2 - 0.5
    out = torch.empty(3, M, N + 1, dtype=torch.float64, device="cuda")
    for k, rows in enumerate((F1, F2, F7)):
        off = 0.0 if k == 0 else 1.0
        v, d1, d2 = U[k, :, 0], U[k, :, 1], U[k, :, 2]
        out[k, :, 0] = mesh.x1 * (d1 - off) + n_rad * (v - off * mesh.x1)
        out[k, :, 1] = mesh.x1 * (d2 - d1) / dx + n_rad * (d1 - off)
        out[k, :, 2:] = rows.view(M, N - 1)
    return out.view(-1)


def _solve_exact(mesh, topo, F):
    """Newton with a dense finite-difference Jacobian."""
    u = _dev(W.flat_guess(mesh))
    eye = torch.eye(u.numel(), dtype=torch.float64, device="cuda")
    for k in range(7):
        Fu = _residual_exact(mesh, topo, F, u)
        if k < 5:
            h = 1e-7
            J = torch.stack([(_residual_exact(mesh, topo, F, u + h * e) - Fu) / h for e in eye], dim=1)
        u = u - torch.linalg.solve(J, Fu)
    return u


def _precond_exact(mesh, F, r, n_rad=0.05):
    """The banded Jacobian of the linearised system (Sec. 4.2, App. B) solved by
    block elimination, half_band slices to a block."""
    N, M, dx, dy = mesh.N, mesh.M, mesh.dx, mesh.dy
    NB, nb = N + 1, 3 * (N + 1)
    h = min(max(1, math.floor(M / 20.0 + 0.5)), M - 1)
    f64 = dict(dtype=torch.float64, device="cuda")
    i = torch.arange(1, N + 1, **f64)
    T = torch.where(i.view(1, -1) < i.view(-1, 1), 1.0, torch.where(i.view(1, -1) == i.view(-1, 1), 0.5, 0.0)).to(torch.float64)
    T[:, 0] = 0.5
    T[0] = 0.0
    Q = torch.cat([torch.ones(N, 1, **f64), dx * T], dim=1)  # nodal values from [q(1), q_x]
    H = 0.5 * (Q[1:] + Q[:-1])
    x, y = mesh.x1 + dx * torch.arange(N, **f64), mesh.y1 + dy * torch.arange(M, **f64)
    s = x.view(1, N) - (x[:-1] + 0.5 * dx).view(-1, 1)
    cx = torch.ones(N, **f64)
    cx[0] = cx[-1] = 0.5
    cy = torch.ones(M, **f64)
    cy[0] = cy[-1] = 0.5
    one, zero = torch.ones(N - 1, **f64), torch.zeros(N - 1, **f64)
    xs = x[:-1] + 0.5 * dx
    E = torch.zeros(N - 1, NB, **f64)
    E[torch.arange(N - 1), torch.arange(1, N)] = 0.5
    E[torch.arange(N - 1), torch.arange(2, N + 1)] = 0.5

    def block(l, m):
        B = torch.zeros(nb, nb, **f64)
        t = float(y[m] - y[l])
        p, w = s * s + t * t, dx * dy * cx * cy[m]
        k5, k7 = torch.rsqrt(p), torch.rsqrt(p + 1)
        B[NB + 2:2 * NB, 1:NB] = w * k5
        B[2 * NB + 2:, 1:NB] = w * k7
        W6 = (w * k7 ** 3) @ Q
        B[NB + 2:2 * NB, 2 * NB:] = W6
        B[2 * NB + 2:, NB:2 * NB] = W6
        if l == m:
            sums = sum((dx * dy * cx * cy[j] * torch.rsqrt(s * s + (y[j] - y[l]) ** 2)).sum(1) for j in range(M))
            sums = sums - _rect(one, zero, one, mesh, xs, y[l].expand(N - 1))
            B[NB + 2:2 * NB, :NB] -= sums.view(-1, 1) * E
            for f in range(3):
                B[f * NB, f * NB], B[f * NB, f * NB + 1] = n_rad, mesh.x1
                B[f * NB + 1, f * NB + 1], B[f * NB + 1, f * NB + 2] = n_rad - mesh.x1 / dx, mesh.x1 / dx
            B[2:NB, :NB] = H / F ** 2
            B[2:NB, NB:2 * NB] = E
            B[NB + 2:2 * NB, NB:2 * NB] -= 2 * math.pi * H
            B[2 * NB + 2:, 2 * NB:] -= 2 * math.pi * H
        return B

    def span(rows, cols):
        B = torch.zeros(len(rows) * nb, len(cols) * nb, **f64)
        for a, l in enumerate(rows):
            for b, m in enumerate(cols):
                if abs(l - m) <= h:
                    B[a * nb:(a + 1) * nb, b * nb:(b + 1) * nb] = block(l, m)
        return B

    groups = [list(range(a, min(M, a + h))) for a in range(0, M, h)]
    R = _dev(r).view(3, M, NB).permute(1, 0, 2).reshape(M, nb)
    ys, Ws = [], []
    for k, gk in enumerate(groups):
        D, v = span(gk, gk), R[gk].reshape(-1, 1)
        if k:
            L = span(gk, groups[k - 1])
            D, v = D - L @ Ws[-1], v - L @ ys[-1]
        U = span(gk, groups[k + 1]) if k + 1 < len(groups) else None
        X = torch.linalg.solve(D, v if U is None else torch.cat([v, U], dim=1))
        ys.append(X[:, :1])
        Ws.append(X[:, 1:])
    zs = [None] * len(groups)
    for k in reversed(range(len(groups))):
        zs[k] = ys[k] if k + 1 == len(groups) else ys[k] - Ws[k] @ zs[k + 1]
    return torch.cat([v.view(-1, nb) for v in zs]).view(M, 3, NB).permute(1, 0, 2).reshape(-1)


def _train_exact(case, seed):
    x, t, p = _train_inputs(case, seed)
    p = _dev(p).requires_grad_(True)
    a = torch.nn.functional.pad(_dev(x).permute(0, 3, 1, 2), (0, 0, 0, 0, 0, 12))
    off = 0
    for k, (cin, cout, dil) in enumerate(LAYERS):
        w = p[off:off + 9 * cin * cout].view(cout, 3, 3, cin).permute(0, 3, 1, 2)
        b = p[off + 9 * cin * cout:off + 9 * cin * cout + cout]
        off += 9 * cin * cout + cout
        z = torch.nn.functional.conv2d(a, w, b, padding=dil, dilation=dil)
        a = torch.nn.functional.silu(z)
    loss = ((z[:, :3] - _dev(t).permute(0, 3, 1, 2)) ** 2).mean()
    loss.backward()
    return {"gradient": p.grad.detach(), "loss": float(loss.detach())}


def exact(case, seed):
    kind = case["kind"]
    if kind == "residual":
        mesh, topo, F, u = _residual_inputs(case, seed)
        return _residual_exact(mesh, topo, F, _dev(u))
    if kind == "solve" and case["N"] * case["M"] <= 400:
        mesh, topo, _ = _solve_inputs(case, seed)
        return _solve_exact(mesh, topo, case["F"])
    if kind == "factor":
        mesh, _, F, r = _factor_inputs(case, seed)
        return _precond_exact(mesh, F, r)
    if kind == "train":
        return _train_exact(case, seed)
    return None  # the large solves have no quick 64-bit counterpart
