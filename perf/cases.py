"""The work that a user of this eigensolver has it do, as cases that can be timed and compared.

The entry points are those of ``paper_1710_07080_gb300``: the operator of the trimmed, shifted and
deflated system (with a handle and without one), the inner solve, the multilevel preconditioner, the
Rayleigh-Ritz step after one expansion, whole solves of one graph, and the batched solve.  Graphs are
those of this repository's configurations and tests (2-D and 3-D grids, R-MAT, random geometric,
Erdos-Renyi, Watts-Strogatz, with or without edge weights); a case fixes its graph, the seed its vectors.

What a mixed-precision inner solve returns holds FP32 accuracy in FP64 storage, and an eigenvector is
known to about (residual bound) / (gap to the next eigenvalue): both are taken as FP32, as a
program does that hands them on.  An eigenvector's sign is free: it is set by the start vector.
"""
import math

import numpy as np
import torch

import paper_1710_07080_gb300 as isira
import synthgraphs

DEV = "cuda"


def listed():
    return [
        # the smallest call: one operator application on the small grid, launches and latency only
        {"name": "apply_f32_grid100x100", "kind": "apply", "family": "grid2d", "nx": 100, "ny": 100, "prec": "f32",
         "c": 0},
        # the FP64 operator on a power-law graph with locked vectors (the R-MAT configuration's operator)
        {"name": "apply_f64_rmat20_c4", "kind": "apply", "family": "rmat", "scale": 20, "prec": "f64", "c": 4},
        # a caller that keeps no handle and allows no allocation, medium sparse random graph
        {"name": "noalloc_f32_ws150k_c3", "kind": "noalloc", "family": "ws", "n": 150_001, "prec": "f32", "c": 3},
        # one V-cycle on an irregular mesh (random geometric graph), as an external Krylov method calls it
        {"name": "precond_f32_rgg1M", "kind": "precond", "family": "rgg", "n": 1_000_003, "prec": "f32"},
        # the inner solve of a power-law graph (diagonal preconditioner), mixed precision
        {"name": "inner_f32_rmat20_c4", "kind": "inner", "family": "rmat", "scale": 20, "prec": "f32", "c": 4,
         "precond": 0},
        # a few iterations of the multilevel-preconditioned inner solve in FP64 on a weighted mesh of ragged size, as
        # an approximate shift-invert step of another eigensolver takes them (in FP32 the same few iterations are
        # known to about 1e-4 only: the whole mixed solves below are what runs them)
        {"name": "inner_f64_wgrid613x487_c3", "kind": "inner", "family": "grid2d", "nx": 613, "ny": 487,
         "weighted": True, "prec": "f64", "c": 3, "precond": 1, "max_it": 8},
        # the inner solve of a small graph, as the batch has hundreds of: latency of the iteration
        {"name": "inner_f32_er12k_c2", "kind": "inner", "family": "er", "n": 12_347, "prec": "f32", "c": 2,
         "precond": 0},
        # Rayleigh-Ritz of a middle-sized search space after one expansion (every outer step)
        {"name": "rayleigh_ritz_k41", "kind": "warm", "k": 41, "w": 40},
        # a whole plain-FP64 solve of a small 2-D grid, the tolerance of the 100 x 100 configuration
        {"name": "solve_f64_grid112x88", "kind": "solve", "family": "grid2d", "nx": 112, "ny": 88, "prec": "f64",
         "pairs": 5, "tol": 1e-10},
        # a whole mixed-precision solve of a large 3-D grid with the solver's own choice of preconditioner
        {"name": "solve_mixed_grid118x109x101", "kind": "solve", "family": "grid3d", "nx": 118, "ny": 109,
         "nz": 101, "prec": "f32", "pairs": 5, "tol": 1e-10},
        # a whole mixed-precision solve of a large power-law graph
        {"name": "solve_mixed_rmat20", "kind": "solve", "family": "rmat", "scale": 20, "prec": "f32", "pairs": 4,
         "tol": 1e-9},
        # many graphs of uneven size at once, the three families of the batched configuration
        {"name": "batch_mixed_12", "kind": "batch", "graphs": 12, "nmin": 1_000, "nmax": 60_000, "pairs": 4,
         "rel_tol": 1e-12},
    ]


# ------------------------------------------------------------------------------------------ drawn cases

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _graph(rng, families, lo, hi):
    """A graph of one of the families with about n vertices, n log-uniform in [lo, hi]."""
    family = rng.choice(families)
    n = _log(rng, lo, hi)
    if family == "grid2d":
        nx = max(3, int(round(math.sqrt(n) * rng.uniform(0.8, 1.6))))
        return {"family": family, "nx": nx, "ny": max(3, n // nx)}
    if family == "grid3d":
        nx = max(3, int(round(n ** (1 / 3) * rng.uniform(0.9, 1.4))))
        ny = max(3, int(round(math.sqrt(n / nx) * rng.uniform(0.9, 1.2))))
        return {"family": family, "nx": nx, "ny": ny, "nz": max(3, n // (nx * ny))}
    if family == "rmat":
        return {"family": family, "scale": max(11, min(20, int(round(math.log2(n)))))}
    return {"family": family, "n": n}


def draw(rng):
    kind = rng.choice(["apply", "noalloc", "precond", "inner", "inner", "inner", "warm", "solve", "solve", "batch"])
    prec = rng.choice(["f32", "f64"])
    if kind == "warm":
        k = rng.randint(4, 64)
        return {"kind": kind, "k": k, "w": k - 1}
    if kind == "apply":
        g = _graph(rng, ["grid2d", "grid3d", "rmat", "rgg", "er", "ws"], 2_000, 600_000)
        return {"kind": kind, **g, "weighted": rng.random() < 0.25, "prec": prec, "c": rng.randint(0, 10)}
    if kind == "noalloc":
        g = _graph(rng, ["grid2d", "rgg", "er", "ws"], 2_000, 600_000)
        return {"kind": kind, **g, "prec": prec, "c": rng.randint(0, 8)}
    if kind == "precond":
        g = _graph(rng, ["grid2d", "grid3d", "rgg"], 5_000, 1_000_000)
        return {"kind": kind, **g, "prec": prec}
    if kind == "inner" and rng.random() < 0.3:
        # mesh-like graphs: the multilevel preconditioner
        g = _graph(rng, ["grid2d", "grid3d", "rgg"], 20_000, 600_000)
        return {"kind": kind, **g, "weighted": rng.random() < 0.25, "prec": "f64", "c": rng.randint(0, 12),
                "precond": 1, "max_it": rng.randint(3, 8)}
    if kind == "inner":
        g = _graph(rng, ["rmat", "er", "ws"], 3_000, 400_000)
        return {"kind": kind, **g, "weighted": rng.random() < 0.25, "prec": prec, "c": rng.randint(0, 12),
                "precond": 0}
    if kind == "solve":
        # simple eigenvalues: with a double one the eigenvectors are not determined
        while True:
            g = _graph(rng, ["grid2d", "grid3d"], 1_000, 12_000 if rng.random() < 0.5 else 150_000)
            pairs = rng.randint(3, 8)
            if _gap(_dims(g), pairs) > 1e-4:
                return {"kind": kind, **g, "prec": prec, "pairs": pairs, "tol": 1e-10}
    return {"kind": kind, "graphs": rng.randint(3, 12), "nmin": 1_000, "nmax": _log(rng, 4_000, 40_000),
            "pairs": rng.randint(2, 4), "rel_tol": 1e-12}


# ------------------------------------------------------------------------------------------ inputs

def _dims(case):
    return [case[d] for d in ("nx", "ny", "nz") if d in case]


def _modes(dims, k):
    """The k smallest positive eigenvalues of a grid and their mode numbers: the Laplacian is the Kronecker
    sum of path Laplacians, whose eigenvalues are 2 - 2 cos(pi i / N)."""
    top = [min(N, k + 2) for N in dims]
    modes = np.stack(np.meshgrid(*[np.arange(t) for t in top], indexing="ij"), -1).reshape(-1, len(dims))
    lam = sum(4.0 * np.sin(np.pi * modes[:, a] / (2 * N)) ** 2 for a, N in enumerate(dims))
    order = np.argsort(lam, kind="stable")[1:k + 1]
    return lam[order], modes[order]


def _gap(dims, k):
    lam, _ = _modes(dims, k + 1)
    return float(np.min(np.diff(lam)))


def _grid_vectors(dims, modes):
    """The unit eigenvectors of the given modes, [n, k] with contiguous columns."""
    cols = []
    for m in modes:
        v = torch.ones(1, dtype=torch.float64, device=DEV)
        for N, i in zip(dims, m):
            x = torch.cos(math.pi * float(i) * (torch.arange(N, dtype=torch.float64, device=DEV) + 0.5) / N)
            v = (v[:, None] * (x / x.norm())[None, :]).reshape(-1)
        cols.append(v)
    return torch.stack(cols).t()


def _grid(dims):
    """CSR of the grid whose vertex (a, b, ...) has the row-major id, columns ascending."""
    n = math.prod(dims)
    idx = torch.arange(n, device=DEV)
    coord, stride, rest = [], [], n
    for N in dims:
        rest //= N
        coord.append(idx // rest % N)
        stride.append(rest)
    down = [(coord[a] > 0, -stride[a]) for a in range(len(dims))]
    up = [(coord[a] < dims[a] - 1, stride[a]) for a in reversed(range(len(dims)))]
    has = torch.stack([h for h, _ in down + up], 1)
    col = torch.stack([idx + d for _, d in down + up], 1)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(has.sum(1), 0)
    return rp, col[has].to(torch.int32)


def _csr(case, seed=1):
    f = case["family"]
    if f in ("grid2d", "grid3d"):
        return _grid(_dims(case))
    if f == "rmat":
        return synthgraphs.rmat_gpu(case["scale"], seed=seed)
    if f == "rgg":
        return synthgraphs.rgg_gpu(case["n"], 12.0, seed=seed)
    make = {"er": lambda: synthgraphs.erdos_renyi(case["n"], 8.0, seed=seed),
            "ws": lambda: synthgraphs.watts_strogatz(case["n"], 10, 0.1, seed=seed)}[f]
    g = make()
    return torch.from_numpy(g.row_ptr).to(DEV), torch.from_numpy(g.col_idx).to(DEV)


def _rows(rp):
    return torch.repeat_interleave(torch.arange(rp.numel() - 1, device=DEV), rp[1:] - rp[:-1])


def _weights(rp, ci):
    """Positive symmetric edge weights in [0.5, 2): a hash of the edge's two ends."""
    u, v = _rows(rp), ci.long()
    a, b = torch.minimum(u, v), torch.maximum(u, v)
    h = (a * 2654435761 + b * 40503 + 12345) % 1000003
    return 0.5 + 1.5 * ((h * 7919) % 1000003).double() / 1000003.0


def _orthonormal(n, c, gen):
    """c orthonormal columns orthogonal to the all-ones vector, laid out as eigpairs() returns them."""
    if c == 0:
        return None
    m = torch.randn(n, c + 1, dtype=torch.float64, device=DEV, generator=gen)
    m[:, 0] = 1.0
    q, _ = torch.linalg.qr(m)
    return q[:, 1:].t().contiguous().t()


def _deflation(case, n, gen):
    """Locked vectors and a shift below the next eigenvalue: a grid's own lowest eigenvectors and the solver's
    rule for the shift, else random orthonormal directions with a small shift."""
    c = case.get("c", 0)
    if case["family"] in ("grid2d", "grid3d") and not case.get("weighted"):
        lam, modes = _modes(_dims(case), c + 1)
        low = lam[c - 1] if c else 0.0
        sigma = lam[c] - max(0.1 * (lam[c] - low), 0.01 * lam[c]) if c else 0.0
        return (_grid_vectors(_dims(case), modes[:c]) if c else None), float(sigma)
    sigma = 2e-5 if case["family"] in ("grid2d", "grid3d", "rgg") else 2e-3
    return _orthonormal(n, c, gen), sigma if c else 0.0


def _unit(n, gen):
    x = torch.randn(n, dtype=torch.float64, device=DEV, generator=gen)
    x -= x.mean()
    return x / x.norm()


def _laplacian(rp, ci, w, n):
    """(weighted degrees, adjacency matrix) in FP64."""
    w = w if w is not None else torch.ones(ci.numel(), dtype=torch.float64, device=DEV)
    A = torch.sparse_csr_tensor(rp, ci.long(), w, size=(n, n), dtype=torch.float64)
    return (A @ torch.ones(n, 1, dtype=torch.float64, device=DEV))[:, 0], A


def _residual(rp, ci, w, n, gen):
    """The residual of an approximate eigenvector, as the inner solve gets it: of a random vector after three
    smoothing steps, scaled to unit norm."""
    d, A = _laplacian(rp, ci, w, n)
    u = _unit(n, gen)
    for _ in range(3):
        u = 0.5 * u + 0.5 * (A @ u[:, None])[:, 0] / d
        u = u - u.mean()
    Lu = d * u - (A @ u[:, None])[:, 0]
    r = Lu - (u @ Lu) / (u @ u) * u
    r = r - r.mean()
    return r / r.norm()


def _batch_graphs(case):
    """Sizes log-spaced over the range; families in turn; grids of aspect 1.27, whose low eigenvalues are simple."""
    out = []
    G = case["graphs"]
    for g in range(G):
        n = int(round(case["nmin"] * (case["nmax"] / case["nmin"]) ** (g / max(1, G - 1))))
        if g % 3 == 1:
            nx = int(round(math.sqrt(1.272 * n)))
            out.append(_grid([nx, max(3, n // nx)]))
        else:
            out.append(_csr({"family": "er" if g % 3 == 0 else "ws", "n": n}, 1000 + g))
    return out


def _problem(case, seed):
    """Graph, weights, vectors and shift of an apply, noalloc, precond or inner case."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    rp, ci = _csr(case)
    n = rp.numel() - 1
    w = _weights(rp, ci) if case.get("weighted") else None
    V, sigma = _deflation(case, n, gen) if case["kind"] != "precond" else (None, 0.0)
    x = _residual(rp, ci, w, n, gen) if case["kind"] == "inner" else _unit(n, gen)
    if case["kind"] == "inner" and V is not None:
        x = x - V @ (V.t() @ x)             # a residual is orthogonal to what is locked
    if case["kind"] in ("apply", "noalloc", "precond") and case["prec"] == "f32":
        x = x.float()
    return {"rp": rp, "ci": ci, "w": w, "V": V, "sigma": sigma, "x": x, "n": n}


def _ritz(case, seed):
    """H = [H0 h; h^T eta] with H0's eigenvectors: Ritz values spread over a Laplacian's spectrum, the low ones
    close to convergence (small couplings)."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    k, w = case["k"], case["w"]
    # no two Ritz values closer than their mean distance on a logarithmic scale allows
    t = torch.arange(w, dtype=torch.float64, device=DEV)
    t = t + 0.6 * torch.rand(w, dtype=torch.float64, device=DEV, generator=gen)
    theta = 1e-3 * torch.exp(t * (math.log(1.2e4) / w))
    q, _ = torch.linalg.qr(torch.randn(w, w, dtype=torch.float64, device=DEV, generator=gen))
    H = torch.zeros(k, k, dtype=torch.float64, device=DEV)
    H[:w, :w] = (q * theta) @ q.t()
    if w < k:
        h = q @ (theta.sqrt() * 0.2 * torch.randn(w, dtype=torch.float64, device=DEV, generator=gen))
        H[:w, w] = h
        H[w, :w] = h
        H[w, w] = 2.0 + torch.rand(1, dtype=torch.float64, device=DEV, generator=gen).item()
    H = 0.5 * (H + H.t())
    _, S0 = torch.linalg.eigh(H[:w, :w])
    return {"H": H, "S0": S0.contiguous()}


# ------------------------------------------------------------------------------------------ the interface

_PREC = {"f32": isira.ISIRA_MIXED, "f64": isira.ISIRA_FP64}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "warm":
        return {"case": case, **_ritz(case, seed)}
    if kind == "batch":
        graphs = _batch_graphs(case)
        gen = torch.Generator(device=DEV).manual_seed(seed)
        return {"case": case, "batch": isira.Batch(graphs, seed=seed % 1000 + 1),
                "towards": [_unit(rp.numel() - 1, gen) for rp, _ in graphs]}
    if kind == "solve":
        gen = torch.Generator(device=DEV).manual_seed(seed)
        rp, ci = _csr(case)
        return {"case": case, "solver": isira.Solver(rp, ci, precision=_PREC[case["prec"]]),
                "u0": _unit(rp.numel() - 1, gen)}
    p = _problem(case, seed)
    if kind == "noalloc":
        deg = p["rp"][1:] - p["rp"][:-1]
        p["trim"] = int(torch.argmax(deg))
        p["delta"] = 2.0 * float(deg.max())
        p["y"] = torch.empty_like(p["x"])
        return {"case": case, **p}
    opts = {"precond": case.get("precond", 1 if kind == "precond" else 0)}
    solver = isira.Solver(p["rp"], p["ci"], weights=p["w"], precision=_PREC[case["prec"]], **opts)
    return {"case": case, "solver": solver, **p}


def _oriented(vec, towards):
    """Eigenvectors with a non-negative product with a given vector, as FP32 coordinates of the vertices."""
    s = torch.sign(towards @ vec)
    return (vec * s).float()


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "warm":
        theta, S, path = isira.sym_eig_warm(state["H"], state["S0"])
        return {"theta": theta, "S": S, "path": path}
    if kind == "apply":
        return state["solver"].apply_operator(state["x"], sigma=state["sigma"], V=state["V"])
    if kind == "noalloc":
        return isira.apply_operator_noalloc(state["rp"], state["ci"], state["x"], state["trim"], sigma=state["sigma"],
                                            delta=state["delta"], V=state["V"], y=state["y"])
    if kind == "precond":
        y, levels, coarsest = state["solver"].precond_apply(state["x"])
        return {"y": y, "levels": levels, "coarsest": coarsest}
    if kind == "inner":
        z, _, _ = state["solver"].inner_solve(state["x"], sigma=state["sigma"], V=state["V"],
                                              max_it=case.get("max_it", 5000), precision=_PREC[case["prec"]])
        return z.float() if case["prec"] == "f32" else z
    if kind == "solve":
        s = state["solver"]
        s.solve(case["pairs"], tol=case["tol"], u0=state["u0"])
        lam, vec, _ = s.eigpairs(want_resid=False)
        return {"eigvals": lam, "embedding": _oriented(vec, state["u0"])}
    b = state["batch"]
    status = b.solve(case["pairs"], rel_tol=case["rel_tol"])
    if status != isira.ISIRA_OK:
        raise RuntimeError(f"batch solve: status {status}")
    out = []
    for g, towards in enumerate(state["towards"]):
        lam, vec, _ = b.eigpairs(g)
        out.append((lam, _oriented(vec, towards)))
    return out


# Iterations that a pass takes, about: the number depends on the graph, not on how an iteration is computed.
_ITERS = {"grid2d": 30, "grid3d": 20, "rgg": 40, "rmat": 10, "er": 10, "ws": 20}


def _shape(case):
    """n and stored entries, about."""
    f = case["family"]
    if f in ("grid2d", "grid3d"):
        d = _dims(case)
        n = math.prod(d)
        return n, 2 * sum(n - n // N for N in d)
    if f == "rmat":
        return int(0.62 * 2 ** case["scale"]), int(30 * 2 ** case["scale"])
    return case["n"], case["n"] * {"rgg": 12, "er": 8, "ws": 10}[f]


def work(case):
    """Inputs once and outputs once; an iterative solve reads the graph and updates its Krylov vectors
    (read z, z_prev, two w, x; write z, w, x) once an iteration."""
    kind = case["kind"]
    if kind == "warm":
        k = case["k"]
        return {"bytes": 8 * (3 * k * k + k), "flops": 2 * k * k * (k + 60)}
    if kind == "batch":
        b = f = 0.0
        for g in range(case["graphs"]):
            n = case["nmin"] * (case["nmax"] / case["nmin"]) ** (g / max(1, case["graphs"] - 1))
            its = 40 * case["pairs"] * (8 if g % 3 == 1 else 1) * 4
            b += its * (4 * 8 * n + 8 * 4 * n)
            f += its * 40 * n
        return {"bytes": b, "flops": f}
    n, nnz = _shape(case)
    word = 4 if case["prec"] == "f32" else 8
    c = case.get("c", 0)
    graph = 4 * nnz + (word * nnz if case.get("weighted") else 0)
    if kind in ("apply", "noalloc"):
        return {"bytes": graph + 8 * n + 2 * word * n + 8 * c * n, "flops": 2 * nnz + (4 + 4 * c) * n}
    if kind == "precond":
        return {"bytes": 2 * graph + 2 * word * n, "flops": 6 * nnz + 12 * n}
    sweeps = 3 if case.get("precond", 0) == 1 or (kind == "solve" and n >= 20_000) else 1
    its = case.get("max_it", _ITERS[case["family"]]) * (8 * case["pairs"] if kind == "solve" else 1) * (6 if kind == "solve" and sweeps == 1 else 1)
    return {"bytes": its * (sweeps * graph + (8 + c) * word * n), "flops": its * (sweeps * 2 * nnz + (30 + 4 * c) * n)}


# ------------------------------------------------------------------------------------------ exact results

def _operator(p):
    """The trimmed operator in FP64: y = (d - sigma) x - A x + (sigma / n) 1^T x + delta V V^T x off the trimmed vertex."""
    n = p["n"]
    d, A = _laplacian(p["rp"], p["ci"], p["w"], n)
    trim = int(torch.nonzero(d == d.max())[0])
    delta = 2.0 * float(d.max())
    V, sigma = p["V"], p["sigma"]
    if V is not None:
        V = V.clone()
        V[trim] = 0.0

    def apply(x):
        x = x.clone()
        x[trim] = 0.0
        y = (d - sigma) * x - (A @ x[:, None])[:, 0] + sigma / n * x.sum()
        if V is not None:
            y = y + delta * (V @ (V.t() @ x))
        y[trim] = 0.0
        return y

    D = torch.maximum(d - sigma, 0.5 * d)
    if V is not None:
        C = torch.linalg.inv(torch.eye(V.shape[1], dtype=torch.float64, device=DEV) / delta + V.t() @ (V / D[:, None]))

    def precond(y):
        z = y / D
        if V is not None:
            z = (y - V @ (C @ (V.t() @ z))) / D
        z[trim] = 0.0
        return z

    return apply, precond, trim


def _minres(apply, precond, b, tau, max_it):
    """Preconditioned MINRES (Paige and Saunders 1975) from x = 0 to the relative preconditioned residual tau."""
    x = torch.zeros_like(b)
    w1, w2 = torch.zeros_like(b), torch.zeros_like(b)
    r1, r2 = torch.zeros_like(b), b.clone()
    y = precond(r2)
    beta = beta1 = math.sqrt(float(r2 @ y))
    oldb, dbar, eps, phibar, cs, sn = 0.0, 0.0, 0.0, beta1, -1.0, 0.0
    for it in range(1, max_it + 1):
        v = y / beta
        y = apply(v)
        if it > 1:
            y = y - (beta / oldb) * r1
        alpha = float(v @ y)
        y = y - (alpha / beta) * r2
        r1, r2 = r2, y
        y = precond(r2)
        oldb, beta = beta, math.sqrt(max(0.0, float(r2 @ y)))
        oldeps, dlt = eps, cs * dbar + sn * alpha
        gbar, eps, dbar = sn * dbar - cs * alpha, sn * beta, -cs * beta
        gamma = math.hypot(gbar, beta)
        cs, sn = gbar / gamma, beta / gamma
        phi, phibar = cs * phibar, sn * phibar
        w = (v - oldeps * w1 - dlt * w2) / gamma
        w1, w2 = w2, w
        x = x + phi * w
        if phibar <= tau * beta1 or not beta > 0.0:
            break
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "warm":
        s = _ritz(case, seed)
        theta, S = torch.linalg.eigh(s["H"])
        big = S.abs().argmax(0)
        S = S * torch.sign(S.gather(0, big[None, :]))
        return {"theta": theta, "S": S, "path": None}
    if kind in ("apply", "noalloc"):
        p = _problem(case, seed)
        apply, _, _ = _operator(p)
        return apply(p["x"].double())
    if kind == "inner" and not case["precond"]:
        p = _problem(case, seed)
        apply, precond, trim = _operator(p)
        b = p["x"].clone()
        b[trim] = 0.0
        x = _minres(apply, precond, b, 1e-3, 5000)
        return x - x.mean()
    if kind == "solve" and case["family"] in ("grid2d", "grid3d"):
        # a grid's eigenpairs in closed form
        gen = torch.Generator(device=DEV).manual_seed(seed)
        lam, modes = _modes(_dims(case), case["pairs"])
        vec = _grid_vectors(_dims(case), modes)
        u0 = _unit(vec.shape[0], gen)
        return {"eigvals": torch.from_numpy(lam), "embedding": vec * torch.sign(u0 @ vec)}
    # the V-cycle's coarse levels come from the framework's own clustering, so a cycle, an inner solve
    # preconditioned by it and a large random graph's eigenpairs have no value from plain torch
    return None
