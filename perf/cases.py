"""Performance cases: the calls a user of the Helmholtz solver makes, over the sizes it is used at.

Every case is a solve of -Delta u - k^2 u = f on (0,1)^d with impedance boundaries, to a
relative FP64 residual ``tol``, through the public entry points:

* ``how = "solve"``: the handle is set up once and kept; a pass is one right-hand side.
* ``how = "oneshot"``: a pass sets the problem up, solves it and releases the handle, as a
  program does that sees each wavenumber or medium once.
* ``how = "batch"``: a pass sets up and solves ``count`` independent problems together.

Results are the whole solution fields.
"""
import math

import numpy as np
import torch

import paper_2512_12538_gb300 as hh

MAX_ITER = 2000


def _case(name, how, n, kh, **more):
    c = {"name": name, "how": how, "dim": 2, "n": n, "kh": kh, "levels": 2, "overlap": 2, "rank": 16,
         "oversample": 10, "precision": "mixed", "outer": "oras", "scheme": "fd", "layers": 0.0, "tol": 1e-10,
         "count": 1}
    c.update(more)
    return c


THREE = {"levels": 3, "overlap": 4, "rank": 32}     # the hierarchy of the larger grids


def listed():
    return [
        # 1D line of 1000 points, two overlapping subdomains, a-harmonic coarse space: the
        # smallest call, all latency (the workload helm1d_n1000_k20pi)
        _case("solve_1d_1000_fp64", "solve", 1000, 20 * math.pi / 1001, dim=1, levels=1, overlap=4, rank=1,
              oversample=0, precision="fp64"),
        # a small 2D problem of the batch configuration's lower end, handle kept: many
        # sources in one medium (an inverse-problem sweep on a coarse grid)
        _case("solve_127_mixed", "solve", 127, 0.3, oversample=8),
        # the 255 x 255, k = 40 workload with its handle kept: many sources, one medium
        _case("solve_255_mixed", "solve", 255, 40.0 / 256),
        # the same workload in the full-precision form
        _case("solve_255_fp64", "solve", 255, 40.0 / 256, precision="fp64"),
        # the 255 x 255 workload solved once: a new wavenumber per call (frequency sweep)
        _case("oneshot_255_mixed", "oneshot", 255, 40.0 / 256),
        # ragged grid, bilinear elements, GMRES (the paper's discretisation and outer solver)
        _case("oneshot_201_q1_gmres", "oneshot", 201, 0.2, outer="gmres", scheme="q1"),
        # layered medium (8 layers, contrast 5), GMRES on explicit-inverse leaves
        _case("oneshot_127_layered", "oneshot", 127, 0.5, outer="gmres", layers=5.0, overlap=4, rank=24,
              oversample=8),
        # a frequency and size mix solved together (the batch configuration)
        _case("batch_48_mixed", "batch", 255, 0.6, oversample=8, count=48),
        # 3-level hierarchy at the middle of its range, ragged, one shot by GMRES
        _case("oneshot_500_gmres", "oneshot", 500, 0.2, outer="gmres", **THREE),
        # the full-precision form on a 3-level hierarchy
        _case("oneshot_383_fp64_gmres", "oneshot", 383, 0.1, outer="gmres", precision="fp64", **THREE),
        # the 1023 x 1023, k = 100 workload: one-shot stationary solve, at the residual that
        # gives relative error 1e-8 with a margin (the benchmark's step)
        _case("oneshot_1023_mixed", "oneshot", 1023, 100.0 / 1024, tol=3e-9, **THREE),
        # the same workload with its handle kept, by GMRES: many sources on the largest grid
        _case("solve_1023_gmres", "solve", 1023, 100.0 / 1024, outer="gmres", **THREE),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    """One more case of these ranges; k h stays where the stationary iteration contracts
    when that is the outer solver."""
    how = rng.choice(("solve", "oneshot"))
    kind = rng.choice(("two", "two", "two_fp64", "two_gmres", "three", "three", "three_fp64", "q1", "layered", "batch",
                       "line"))
    if kind in ("two", "two_fp64"):
        c = _case("", how, _log(rng, 96, 255), rng.uniform(0.15, 0.35), oversample=rng.choice((8, 10)))
        if kind == "two_fp64":
            c["precision"] = "fp64"
    elif kind == "two_gmres":
        c = _case("", how, _log(rng, 63, 255), rng.uniform(0.1, 0.6), outer="gmres")
    elif kind == "three":
        n = _log(rng, 191, 900)
        c = _case("", "solve" if n > 640 else how, n, rng.uniform(0.1, 0.4), outer="gmres", **THREE)
    elif kind == "three_fp64":
        c = _case("", how, _log(rng, 191, 420), rng.uniform(0.1, 0.3), outer="gmres", precision="fp64", **THREE)
    elif kind == "q1":
        c = _case("", how, _log(rng, 63, 255), rng.uniform(0.1, 0.4), outer="gmres", scheme="q1")
    elif kind == "layered":
        c = _case("", how, _log(rng, 63, 160), 0.5, outer="gmres", layers=rng.uniform(1.5, 5.0), overlap=4, rank=24,
                  oversample=8)
    elif kind == "batch":
        c = _case("", "batch", 255, rng.uniform(0.4, 0.6), oversample=8, count=_log(rng, 4, 40))
    else:
        c = _case("", "solve", _log(rng, 400, 4000), rng.uniform(0.02, 0.1), dim=1, levels=1, overlap=4, rank=1,
                  oversample=0, precision="fp64")
    c.pop("name")
    return c


def _problems(case, seed):
    """(n, k) of each problem of a case: one, or the mix of a batch."""
    if case["how"] != "batch":
        return [(case["n"], case["kh"] * (case["n"] + 1))]
    rng = np.random.default_rng(1000 + case["count"])        # the mix belongs to the case
    n = rng.choice((63, 127, 191, 255), case["count"])
    return [(int(m), float(rng.uniform(0.3, case["kh"]) * (m + 1))) for m in n]


def _krows(case, n, k):
    """Wavenumber of each grid row of a medium of 8 horizontal layers, speeds 1 and c0
    alternating; a row on a layer boundary takes the mean of k^2 over its two layers."""
    if not case["layers"]:
        return None
    y = np.arange(n + 2) * (8.0 / (n + 1))
    kl = k / np.where(np.arange(8) % 2 == 0, 1.0, case["layers"])
    lo = np.clip(np.ceil(y - 1e-9).astype(int) - 1, 0, 7)
    hi = np.clip(np.floor(y + 1e-9).astype(int), 0, 7)
    return np.sqrt(0.5 * (kl[lo] ** 2 + kl[hi] ** 2))


def _inputs(case, n, k, rng):
    """Eight point sources of width 2 h, and an incident plane wave on the boundary."""
    S, h = n + 2, 1.0 / (n + 1)
    if case["dim"] == 1:
        f = rng.standard_normal((S, 2)) @ np.array([1.0, 1j])
        g = rng.standard_normal((2, 2)) @ np.array([1.0, 1j])
        return torch.from_numpy(f.reshape(S, 1)).cuda(), torch.from_numpy(g).cuda()
    x = torch.arange(S, dtype=torch.float64, device="cuda") * h
    amp = torch.from_numpy(rng.standard_normal((8, 2)) @ np.array([1.0, 1j])).cuda()
    ctr = torch.from_numpy(rng.uniform(0.0, 1.0, (2, 8, 1))).cuda()
    gx, gy = (torch.exp(-(x[None, :] - c) ** 2 / (8.0 * h * h)) for c in ctr)
    f = (gy.to(torch.complex128) * amp[:, None]).T @ gx.to(torch.complex128)
    t = rng.uniform(0.0, 2.0 * math.pi)
    a, kx, ky = 0.1, k * math.cos(t), k * math.sin(t)
    ex, ey = torch.exp(1j * kx * x), torch.exp(1j * ky * x)
    g = a * torch.stack([1j * (-kx - k) * ey, 1j * (kx - k) * ey * ex[-1], 1j * (-ky - k) * ex,
                         1j * (ky - k) * ex * ey[-1]])
    return f.contiguous(), g.contiguous()


def _options(case, n, k):
    o = {"dim": case["dim"], "n": n, "k": k, "levels": case["levels"], "overlap": case["overlap"],
         "rank": case["rank"], "oversample": case["oversample"], "tol": case["tol"], "max_iter": MAX_ITER,
         "precision": case["precision"], "outer": case["outer"], "seed": 1}
    if case["scheme"] == "q1":
        o["flags"] = hh.HH_FLAG_BILINEAR
    if case["layers"]:
        o.update(k_rows=_krows(case, n, k), leaf_solver="block")
    return o


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    probs = _problems(case, seed)
    state = {"how": case["how"], "options": [_options(case, n, k) for n, k in probs],
             "inputs": [_inputs(case, n, k, rng) for n, k in probs]}
    if case["how"] == "solve":
        state["solver"] = hh.Solver(**state["options"][0])
    return state


def run(state):
    if state["how"] == "batch":
        handles = hh.hh_setup_batch([hh.make_params(**o) for o in state["options"]])
        fs, gs = zip(*state["inputs"])
        us = [torch.empty_like(f) for f in fs]
        hh.hh_solve_batch(handles, fs, gs, us)
        for h in handles:
            hh.hh_destroy(h)
        return us
    f, g = state["inputs"][0]
    if state["how"] == "solve":
        return state["solver"].solve(f, g)[0]
    solver = hh.Solver(**state["options"][0])
    u = solver.solve(f, g)[0]
    solver.close()
    return u


def work(case):
    """Sources and boundary data read once, the solution written once, and its residual
    formed once (a 5- or 9-point row: the test that ends every solve)."""
    by = fl = 0.0
    for n, _ in _problems(case, 0):
        S = n + 2
        pts = S if case["dim"] == 1 else S * S
        by += 16.0 * (2 * pts + (2 if case["dim"] == 1 else 4 * S))
        fl += (8.0 * 9 if case["scheme"] == "q1" else 20.0) * pts
    return {"bytes": by, "flops": fl}


def _line(S, scheme):
    """1D stiffness over h (dense), mass over h and end flags on S nodes."""
    X = 2.0 * np.eye(S) - np.eye(S, k=1) - np.eye(S, k=-1)
    X[0, 0] = X[-1, -1] = 1.0
    b = np.zeros(S)
    b[0] = b[-1] = 1.0
    M = np.eye(S)
    M[0, 0] = M[-1, -1] = 0.5
    if scheme == "q1":
        M = (4.0 * np.eye(S) + np.eye(S, k=1) + np.eye(S, k=-1)) / 6.0
        M[0, 0] = M[-1, -1] = 2.0 / 6.0
    return X, M, np.diag(b)


def _exact2d(case, n, k, f, g):
    S, h = n + 2, 1.0 / (n + 1)
    X, M, E = _line(S, case["scheme"])
    rhs = h * h * (M @ f @ M)
    rhs[:, 0] += h * (M @ g[0])
    rhs[:, -1] += h * (M @ g[1])
    rhs[0, :] += h * (M @ g[2])
    rhs[-1, :] += h * (M @ g[3])
    kr = _krows(case, n, k)
    if kr is None:
        # A U = M U Kx + Ky U M with Ky = X - i kh E, Kx = Ky - (kh)^2 M: diagonal in the
        # eigenvectors of the pencil (Ky, M), with two steps of refinement
        q = k * h
        Ky = X - 1j * q * E
        Kx = Ky - q * q * M
        mu, V = np.linalg.eig(np.linalg.solve(M, Ky))
        L = np.linalg.inv(M @ V)
        den = mu[:, None] + mu[None, :] - q * q
        u = np.zeros((S, S), dtype=np.complex128)
        for _ in range(3):
            r = rhs - (M @ u) @ Kx - (Ky @ u) @ M
            u = u + V @ ((L @ r @ L.T) / den) @ V.T
        return u
    # layered: block elimination over the grid rows (blocks of one row)
    q, w = kr * h, np.diag(M).copy()
    off = -np.diag(w).astype(np.complex128)
    inv, y = [], []
    for j in range(S):
        D = w[j] * (X - q[j] ** 2 * M - 1j * q[j] * E) + (X[j, j] - 1j * q[j] * E[j, j]) * M
        v = rhs[j]
        if j:
            D = D - off @ inv[-1] @ off
            v = v - off @ (inv[-1] @ y[-1])
        inv.append(np.linalg.inv(D))
        y.append(v)
    u = np.zeros((S, S), dtype=np.complex128)
    for j in range(S - 1, -1, -1):
        u[j] = inv[j] @ (y[j] if j == S - 1 else y[j] - off @ u[j + 1])
    return u


def _exact1d(n, k, f, g):
    S, h = n + 2, 1.0 / (n + 1)
    X, M, E = _line(S, "fd")
    rhs = h * h * (M @ f[:, 0])
    rhs[0] += h * g[0]
    rhs[-1] += h * g[1]
    q = k * h
    return np.linalg.solve(X - q * q * M - 1j * q * E, rhs).reshape(S, 1)


def exact(case, seed):
    """The solution of the discrete system by plain numpy in 64 bits."""
    rng = np.random.default_rng(seed)
    out = []
    for n, k in _problems(case, seed):
        f, g = (t.cpu().numpy() for t in _inputs(case, n, k, rng))
        out.append(_exact1d(n, k, f, g) if case["dim"] == 1 else _exact2d(case, n, k, f, g))
    return out if case["how"] == "batch" else out[0]
