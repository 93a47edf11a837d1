"""What a user of this library has it do, as timed cases.

Kinds (field "kind"), each one call or a short sequence of calls of the public
Python API over libamg.so:

* cycle    -- Hierarchy.precond_apply: one V(1,1) cycle z = M r, the building
              block a program with its own Krylov loop calls;
* solve    -- Hierarchy.solve: PCG or GMRES to 1e-8 on a hierarchy set up before;
* adaptive -- Hierarchy.sparsify back to gamma = 1, then Hierarchy.solve with
              adaptive=True (Algorithm 5: reintroduction on slow convergence);
* batch    -- Hierarchy.solve_batch: k right-hand sides through one hierarchy;
* step     -- Hierarchy.setup and Hierarchy.solve: a new matrix every time step;
* serve    -- Server.submit / wait of a burst of requests on two hierarchies.

Fields: "grid" (2d5: 2D 5-point, 3d7: 3D 7-point, 3d27: 3D 27-point, fv7: 3D
finite volumes with lognormal coefficients, aniso: rotated anisotropic Q1),
"N" (points per side), "precision" (fp64, fp32, bf16: the cycle's storage;
Krylov loops are FP64), "gamma" (drop tolerance of every coarse level), and
per kind "krylov", "lump", "k", "host" (host arrays in and out).  Matrices,
coefficients and right-hand sides are made on the GPU, the random ones from
the seed (right-hand sides uniform in [-1, 1), as in the benchmark).
"""
import math

import numpy as np
import torch

from paper_1512_04629_gb300 import Hierarchy
from paper_1512_04629_gb300.amg import (KRYLOV_CG, KRYLOV_GMRES, LUMP_DIAG, LUMP_STRONG, PREC_FP32, PREC_FP32_BF16,
                                        PREC_FP64, Server, csr_struct)

TOL = 1e-8
PRECISION = {"fp64": PREC_FP64, "fp32": PREC_FP32, "bf16": PREC_FP32_BF16}
ENTRIES = {"2d5": 5, "3d7": 7, "3d27": 27, "fv7": 7, "aniso": 9}  # stored entries of an interior row


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a 64 x 64 grid's cycle, 16 short kernels one after another
        {"name": "cycle_2d5_64", "kind": "cycle", "grid": "2d5", "N": 64, "precision": "fp64", "gamma": 0.1},
        # the benchmark's operator, 2.1 M unknowns, in double precision
        {"name": "cycle_3d7_128", "kind": "cycle", "grid": "3d7", "N": 128, "precision": "fp64", "gamma": 0.1},
        # the mixed-precision workload: 27 entries a row, 7.1 M unknowns
        {"name": "solve_3d27_192_bf16", "kind": "solve", "grid": "3d27", "N": 192, "precision": "bf16", "gamma": 0.1,
         "krylov": "cg", "lump": "diag", "host": False},
        # one small system from host memory: latency
        {"name": "solve_2d5_64_host", "kind": "solve", "grid": "2d5", "N": 64, "precision": "fp64", "gamma": 0.1,
         "krylov": "cg", "lump": "diag", "host": True},
        # the benchmark's solve phase
        {"name": "solve_3d7_128", "kind": "solve", "grid": "3d7", "N": 128, "precision": "fp64", "gamma": 0.1,
         "krylov": "cg", "lump": "diag", "host": False},
        # heterogeneous coefficients on an odd grid, FP32 cycle under flexible CG
        {"name": "solve_fv7_101_fp32", "kind": "solve", "grid": "fv7", "N": 101, "precision": "fp32", "gamma": 0.1,
         "krylov": "cg", "lump": "diag", "host": False},
        # full lumping, whose operators may be indefinite, is solved with GMRES
        {"name": "gmres_3d7_96_lump", "kind": "solve", "grid": "3d7", "N": 96, "precision": "fp64", "gamma": 1.0,
         "krylov": "gmres", "lump": "strong", "host": False},
        # too much dropped: entries come back while it solves
        {"name": "adaptive_3d7_75", "kind": "adaptive", "grid": "3d7", "N": 75, "precision": "fp64", "gamma": 1.0},
        # many right-hand sides of one heterogeneous problem
        {"name": "batch_fv7_112_k32_fp32", "kind": "batch", "grid": "fv7", "N": 112, "precision": "fp32",
         "gamma": 0.1, "k": 32},
        # the benchmark's whole step: setup, sparsification and solve
        {"name": "step_3d7_128", "kind": "step", "grid": "3d7", "N": 128, "precision": "fp64", "gamma": 0.1,
         "host": False},
        # the same for a small system in host memory, sizes that divide nothing
        {"name": "step_2d5_101_host", "kind": "step", "grid": "2d5", "N": 101, "precision": "fp64", "gamma": 0.1,
         "host": True},
        # a burst of 24 requests to a server that holds two models
        {"name": "serve_24", "kind": "serve", "grid": "3d7", "N": 48, "precision": "fp32", "gamma": 0.1, "k": 24},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# side lengths drawn per kind: (2D, 3D, 27-point) upper ends
_SIDES = {"cycle": (1400, 150, 150), "solve": (1000, 120, 96), "adaptive": (400, 75, 56), "batch": (512, 96, 64),
          "step": (900, 110, 80), "serve": (160, 48, 40)}


def draw(rng):
    kind = rng.choice(["cycle", "cycle", "solve", "solve", "adaptive", "batch", "batch", "step", "step", "serve"])
    grid = rng.choice(["2d5", "3d7", "3d27", "fv7", "aniso"] if kind in ("cycle", "step") else
                      ["2d5", "3d7", "3d27"] if kind == "adaptive" else ["2d5", "3d7", "3d27", "fv7"])
    top = _SIDES[kind]
    if grid in ("2d5", "aniso"):
        N = _log_int(rng, 40, top[0] if grid == "2d5" else min(top[0], 400))
    else:
        N = _log_int(rng, 14, top[2] if grid == "3d27" else top[1])
    case = {"kind": kind, "grid": grid, "N": N, "precision": rng.choice(["fp64", "fp64", "fp32", "bf16"]),
            "gamma": rng.choice([0.0, 0.01, 0.1])}
    if kind == "cycle":
        case["precision"] = "fp64"
    if kind == "solve":
        gmres = rng.random() < 0.35
        case.update(krylov="gmres" if gmres else "cg", lump="strong" if gmres and rng.random() < 0.7 else "diag",
                    host=rng.random() < 0.3)
        if case["lump"] == "strong":
            case["gamma"] = rng.choice([0.1, 1.0])
    elif kind == "adaptive":
        case.update(gamma=1.0, precision="fp64")
    elif kind == "batch":
        case["k"] = rng.randint(1, 48)
        case["precision"] = rng.choice(["fp64", "fp32", "fp32"])
    elif kind == "step":
        case["host"] = rng.random() < 0.4
    elif kind == "serve":
        case["k"] = rng.randint(4, 32)
        case["precision"] = "fp32"
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + salt)
    return g


def _rhs(case, seed, k):
    """k right-hand sides, n x k, uniform in [-1, 1)."""
    n = _unknowns(case)
    b = torch.rand(n, k, generator=_gen(seed, 1), device="cuda", dtype=torch.float64)
    return b.mul_(2.0).sub_(1.0)


def _coefficients(N, seed):
    """Cell coefficients exp(2 z), z standard normal."""
    return torch.randn(N, N, N, generator=_gen(seed, 2), device="cuda", dtype=torch.float64).mul_(2.0).exp_()


def _transmissibilities(k):
    """Face transmissibilities of the finite-volume operator, one tensor per
    neighbour (-z, -y, -x, +x, +y, +z): harmonic means inside, 2 k on the
    boundary."""
    out = {}
    for d in range(3):
        a, b = k.narrow(d, 0, k.shape[d] - 1), k.narrow(d, 1, k.shape[d] - 1)
        t = 2.0 * a * b / (a + b)
        lo, hi = (2.0 * k).clone(), (2.0 * k).clone()
        lo.narrow(d, 1, k.shape[d] - 1).copy_(t)
        hi.narrow(d, 0, k.shape[d] - 1).copy_(t)
        out[d, -1], out[d, 1] = lo, hi
    return out


def _aniso_stencil():
    """9-point Q1 stencil of rotated anisotropic diffusion (angle pi / 8, ratio 1e-3)."""
    t, eps = math.pi / 8, 1e-3
    q = np.array([[math.cos(t), math.sin(t)], [-math.sin(t), math.cos(t)]])
    K = q.T @ np.diag([1.0, eps]) @ q
    g = [0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)]
    Ke = np.zeros((4, 4))
    for x in g:
        for y in g:
            G = np.array([[-(1 - y), -(1 - x)], [1 - y, -x], [-y, 1 - x], [y, x]])
            Ke += 0.25 * G @ K @ G.T
    node = {(0, 0): 0, (1, 0): 1, (0, 1): 2, (1, 1): 3}
    st = {}
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            v = 0.0
            for ey in (0, 1):
                for ex in (0, 1):
                    c, m = (1 - ex, 1 - ey), (1 - ex + dx, 1 - ey + dy)
                    if m in node:
                        v += Ke[node[c], node[m]]
            st[0, dy, dx] = v
    return st


def _stencil(grid):
    """{(dz, dy, dx): coefficient} of a constant-coefficient operator."""
    if grid == "aniso":
        return _aniso_stencil()
    off = (-1, 0, 1)
    if grid == "3d27":
        return {(z, y, x): 26.0 if (z, y, x) == (0, 0, 0) else -1.0 for z in off for y in off for x in off}
    zs = (0,) if grid == "2d5" else off
    return {(z, y, x): (4.0 if grid == "2d5" else 6.0) if (z, y, x) == (0, 0, 0) else -1.0
            for z in zs for y in off for x in off if abs(z) + abs(y) + abs(x) <= 1}


def _unknowns(case):
    return case["N"] ** (2 if case["grid"] in ("2d5", "aniso") else 3)


def _matrix(grid, N, seed):
    """(rowptr, col, val) CUDA tensors of the operator, rows sorted by column."""
    dims = (1, N, N) if grid in ("2d5", "aniso") else (N, N, N)
    n = dims[0] * N * N
    i = torch.arange(n, device="cuda")
    at = (i // (N * N), (i // N) % N, i % N)
    if grid == "fv7":
        t = _transmissibilities(_coefficients(N, seed))
        diag = sum(t.values()).reshape(-1)
        st = {(0, 0, 0): diag}
        for (d, side), f in t.items():
            st[tuple(side if e == d else 0 for e in range(3))] = -f.reshape(-1)
    else:
        st = _stencil(grid)
    pts = sorted(st)  # lexicographic (dz, dy, dx): increasing columns
    cols = torch.empty(n, len(pts), device="cuda", dtype=torch.int32)
    vals = torch.empty(n, len(pts), device="cuda", dtype=torch.float64)
    mask = torch.empty(n, len(pts), device="cuda", dtype=torch.bool)
    for s, p in enumerate(pts):
        ok = torch.ones(n, device="cuda", dtype=torch.bool)
        for d in range(3):
            if p[d]:
                ok &= (at[d] + p[d] >= 0) & (at[d] + p[d] < dims[d])
        mask[:, s] = ok
        cols[:, s] = (i + (p[0] * N + p[1]) * N + p[2]).to(torch.int32)
        vals[:, s] = st[p]
    rowptr = torch.zeros(n + 1, device="cuda", dtype=torch.int32)
    rowptr[1:] = mask.sum(1).cumsum(0).to(torch.int32)
    return rowptr, cols[mask], vals[mask]


def _options(case):
    return dict(gamma=[0.0, case["gamma"]], precision=PRECISION[case["precision"]],
                krylov=KRYLOV_GMRES if case.get("krylov") == "gmres" or case["grid"] == "aniso" else KRYLOV_CG,
                lump=LUMP_STRONG if case.get("lump") == "strong" else LUMP_DIAG)


def prepare(case, seed):
    kind, grid, N = case["kind"], case["grid"], case["N"]
    s = {"case": case, "kind": kind, "options": _options(case)}
    if kind == "serve":
        # half of the requests go to the operator itself, half to a lognormal one
        grids = [(grid, N), ("fv7", 40)]
        s["server"] = Server(max_batch=8)
        s["hids"] = [s["server"].register(Hierarchy.setup(csr_struct(*_matrix(g, m, seed)), **s["options"]))
                     for g, m in grids]
        s["b"] = []
        for r in range(case["k"]):
            g, m = grids[r % 2]
            b = _rhs({"grid": g, "N": m}, seed + 7919 * (r + 1), 1)
            s["b"].append((r % 2, b.reshape(-1).cpu().numpy()))
        return s
    A = _matrix(grid, N, seed)
    b = _rhs(case, seed, case.get("k", 1))
    s["b"] = b if kind == "batch" else b.reshape(-1)
    if case.get("host"):
        s["b"] = s["b"].cpu().numpy()
        A = tuple(t.cpu().numpy() for t in A) if kind == "step" else A
    if kind == "step":
        s["A"] = csr_struct(*A)
    else:
        s["h"] = Hierarchy.setup(csr_struct(*A), **s["options"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "cycle":
        z = torch.empty_like(s["b"])
        s["h"].precond_apply(s["b"], z)
        return {"z": z}
    if kind == "serve":
        tickets = [(s["server"].submit(s["hids"][w], b, tol=TOL), s["hids"][w]) for w, b in s["b"]]
        got = [s["server"].wait(t, hid) for t, hid in tickets]
        return {"x": [x for _, x, _ in got], "iterations": np.array([i.iterations for _, _, i in got])}
    if kind == "batch":
        x, info = s["h"].solve_batch(s["b"], tol=TOL)
        return {"x": x, "iterations": np.array([i.iterations for i in info])}
    if kind == "adaptive":
        s["h"].sparsify(s["options"]["gamma"])
        x, info = s["h"].solve(s["b"], tol=TOL, adaptive=True)
        return {"x": x, "iterations": info.iterations, "resets": info.resets}
    h = Hierarchy.setup(s["A"], **s["options"]) if kind == "step" else s["h"]
    x, info = h.solve(s["b"], tol=TOL)
    return {"x": x, "iterations": info.iterations}


# ---------------------------------------------------------------------------
# the least work and the exact results
# ---------------------------------------------------------------------------
def work(case):
    """Each right-hand side read once and each result written once; the
    operator's entries read once where they are data (the CSR arrays that a
    step's setup is given, lognormal coefficients) -- the other operators are a
    stencil's few numbers; and the multiplications by the operator that no
    cycle (two relaxations) and no Krylov solve (one) can leave out."""
    n, k = _unknowns(case), case.get("k", 1)
    nnz = n * ENTRIES[case["grid"]]
    operator = 12 * nnz if case["kind"] == "step" else 8 * nnz if case["grid"] == "fv7" else 0
    return {"bytes": operator + 16 * n * k, "flops": (4 if case["kind"] == "cycle" else 2) * nnz * k}


def _sine_solve(grid, N, b):
    """A^-1 b for the 5-, 7- and 27-point operators, diagonal in the sine basis."""
    j = torch.arange(1, N + 1, device="cuda", dtype=torch.float64)
    S = torch.sin(math.pi / (N + 1) * torch.outer(j, j)) * math.sqrt(2.0 / (N + 1))
    c = torch.cos(math.pi * j / (N + 1))
    if grid == "2d5":
        lam = (2 - 2 * c)[:, None] + (2 - 2 * c)[None, :]
        return (S @ ((S @ b.reshape(N, N) @ S) / lam) @ S).reshape(-1)
    if grid == "3d7":
        e = 2 - 2 * c
        lam = e[:, None, None] + e[None, :, None] + e[None, None, :]
    else:
        e = 1 + 2 * c
        lam = 27 - e[:, None, None] * e[None, :, None] * e[None, None, :]

    def sines(u):
        u = torch.einsum("ai,ijk->ajk", S, u)
        u = torch.einsum("bj,ajk->abk", S, u)
        return torch.einsum("ck,abk->abc", S, u)

    return sines(sines(b.reshape(N, N, N)) / lam).reshape(-1)


def _volume_solve(N, seed, B):
    """A^-1 B (n x k) for the finite-volume operator: Jacobi-preconditioned CG
    down to rounding, by faces on the grid."""
    t = _transmissibilities(_coefficients(N, seed))
    diag = sum(t.values())
    inner = [t[d, 1].narrow(d, 0, N - 1) for d in range(3)]

    def apply(u):
        out = u * diag
        for d in range(3):
            out.narrow(d + 1, 0, N - 1).sub_(inner[d] * u.narrow(d + 1, 1, N - 1))
            out.narrow(d + 1, 1, N - 1).sub_(inner[d] * u.narrow(d + 1, 0, N - 1))
        return out

    r = B.t().reshape(-1, N, N, N).clone()
    dot = lambda u, v: (u * v).sum((1, 2, 3), keepdim=True)  # noqa: E731
    x = torch.zeros_like(r)
    stop = 1e-28 * dot(r, r)
    p = r / diag
    rho = dot(r, p)
    for it in range(20000):
        q = apply(p)
        a = rho / dot(p, q).clamp_min(1e-300)
        x.addcmul_(a, p)
        r.addcmul_(-a, q)
        if it % 50 == 49 and bool((dot(r, r) <= stop).all()):
            break
        z = r / diag
        new = dot(r, z)
        p.mul_(new / rho.clamp_min(1e-300)).add_(z)
        rho = new
    return x.reshape(x.shape[0], -1).t().contiguous()


def exact(case, seed):
    kind, grid, N = case["kind"], case["grid"], case["N"]
    if kind == "cycle" or grid == "aniso":
        return None  # the cycle is defined by the hierarchy that the library builds; no closed form for aniso

    def solution(g, m, B):
        if g == "fv7":
            return _volume_solve(m, seed, B)
        return torch.stack([_sine_solve(g, m, B[:, c].contiguous()) for c in range(B.shape[1])], 1)

    if kind == "serve":
        x = []
        for r in range(case["k"]):
            g, m = (grid, N) if r % 2 == 0 else ("fv7", 40)
            x.append(solution(g, m, _rhs({"grid": g, "N": m}, seed + 7919 * (r + 1), 1)).reshape(-1))
        return {"x": x, "iterations": None}
    X = solution(grid, N, _rhs(case, seed, case.get("k", 1)))
    out = {"x": X if kind == "batch" else X.reshape(-1), "iterations": None}
    if kind == "adaptive":
        out["resets"] = None
    return out
