"""The solver calls whose time is measured, and what they have to give.

Every case is a whole call that a program makes on a hierarchy it holds: a PCG
solve (`Solver.solve`), several right-hand sides (`Solver.solve_multi`),
several meshes (`vasmg_solve_batch`), a solve after new material data
(`Solver.update`), and a request on a mesh not seen before (setup, solve,
release, as a server slot does).  The sizes are the benchmark's four workloads,
the mesh sizes of the tests, and sizes between them.

The solves run to 1e-8, as the smoke run and several tests do: a converged
solution hardly depends on the rounding inside the preconditioner, so what
comes back can be compared closely and against a reference in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2505_09064_gb300 import vasmg

TOL = 1e-8

# ------------------------------------------------------------------ cases


def listed():
    return [
        # The smallest benchmark workload (64 x 64, plain FP64): one launch per
        # iteration does the whole V-cycle, so latency is what counts.
        dict(name="square64_fp64", kind="solve", dim=2, n=64, precision="fp64", nu=0.3, material="plain", graded=1.0, k=1),
        # A small 3D request (14.7k dofs): all levels below the region launches.
        dict(name="cube17_fp32", kind="solve", dim=3, n=17, precision="fp32", nu=0.35, material="plain", graded=1.0, k=1),
        # An ordinary 2D problem of the paper's sizes (about 150k vertices), odd side.
        dict(name="square389_fp32", kind="solve", dim=2, n=389, precision="fp32", nu=0.3, material="plain", graded=1.0, k=1),
        # The large 2D benchmark workload: 1:100 material jumps, FP32 V-cycle.
        dict(name="square1024_checker_fp32", kind="solve", dim=2, n=1024, precision="fp32", nu=0.3, material="checker", graded=1.0, k=1),
        # The ordinary 3D benchmark workload.
        dict(name="cube64_fp32", kind="solve", dim=3, n=64, precision="fp32", nu=0.3, material="plain", graded=1.0, k=1),
        # The plain FP64 path in 3D at the size of the region-launch tests.
        dict(name="cube41_fp64", kind="solve", dim=3, n=41, precision="fp64", nu=0.3, material="plain", graded=1.0, k=1),
        # The headline workload: 6.3M dofs, graded, nearly incompressible, BF16 operator values.
        dict(name="cube128_graded_bf16", kind="solve", dim=3, n=128, precision="bf16", nu=0.45, material="plain", graded=16.0, k=1),
        # Eight load cases on one 3D hierarchy (the most one pass takes).
        dict(name="cube56_graded_bf16_rhs8", kind="multi", dim=3, n=56, precision="bf16", nu=0.45, material="plain", graded=16.0, k=8),
        # Three load cases in 2D: a pass of four with one slot empty.
        dict(name="square257_checker_fp32_rhs3", kind="multi", dim=2, n=257, precision="fp32", nu=0.3, material="checker", graded=1.0, k=3),
        # Six uneven 2D and 3D meshes solved together, as a batching server does.
        dict(name="batch6_fp32", kind="batch", dim=0, n=181, precision="fp32", nu=0.3, material="plain", graded=1.0, k=6),
        # A step of a program whose material changes: new Lame parameters, then a solve.
        dict(name="cube33_update_fp32", kind="update", dim=3, n=33, precision="fp32", nu=0.3, material="random", graded=1.0, k=1),
        # A request on a new mesh: setup, one solve, release.
        dict(name="square220_request_fp32", kind="request", dim=2, n=220, precision="fp32", nu=0.3, material="plain", graded=1.0, k=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "multi", "batch", "update", "request"])
    dim = rng.choice([2, 3])
    # the side ranges keep a drawn case below the headline workload's cost
    if kind in ("solve", "update"):
        n = _log_int(rng, 33, 900) if dim == 2 else _log_int(rng, 9, 88)
    elif kind == "multi":
        n = _log_int(rng, 33, 420) if dim == 2 else _log_int(rng, 9, 52)
    elif kind == "request":
        n = _log_int(rng, 64, 420) if dim == 2 else _log_int(rng, 16, 52)
    else:
        dim, n = 0, _log_int(rng, 64, 320)
    precision = rng.choice(["fp64", "fp32", "fp32", "bf16"]) if kind == "solve" else rng.choice(["fp32", "fp32", "bf16"])
    k = rng.randint(2, 8) if kind == "multi" else (rng.randint(3, 8) if kind == "batch" else 1)
    return dict(kind=kind, dim=dim, n=n, precision=precision, nu=round(rng.uniform(0.2, 0.45), 3),
                material=rng.choice(["plain", "checker", "random"]),
                graded=rng.choice([1.0, 1.0, 16.0]) if dim == 3 else 1.0, k=k)


# ------------------------------------------------------------------ problems

_PERMS = [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]


def _mesh(dim, n, graded, rng):
    """An n^dim vertex grid on the unit square / cube: interior vertices
    jittered (0.2 h in 2D, 0.15 h in 3D) unless graded, quads split along random
    diagonals, hexes into six Kuhn tetrahedra."""
    if graded != 1.0:
        r = graded ** (1.0 / max(1, n - 2))
        t = (r ** np.arange(n) - 1.0) / (r ** (n - 1) - 1.0)
        t[-1] = 1.0
    else:
        t = np.linspace(0.0, 1.0, n)
    axes = np.meshgrid(*([t] * dim), indexing="ij")[::-1]  # x fastest
    coords = np.stack([a.ravel() for a in axes], axis=1)
    if graded == 1.0:
        inner = ((coords > 0.0) & (coords < 1.0)).all(axis=1)
        amp = (0.2 if dim == 2 else 0.15) / (n - 1)
        coords = coords + rng.uniform(-amp, amp, size=coords.shape) * inner[:, None]
    if dim == 2:
        v = (np.arange(n - 1, dtype=np.int32)[:, None] * n + np.arange(n - 1, dtype=np.int32)[None, :]).ravel()
        d = rng.random(v.size) < 0.5
        e = np.empty((v.size, 2, 3), np.int32)
        e[:, 0, 0], e[:, 0, 1], e[:, 0, 2] = v, v + 1, np.where(d, v + n + 1, v + n)
        e[:, 1, 0], e[:, 1, 1], e[:, 1, 2] = np.where(d, v, v + 1), v + n + 1, v + n
        return np.ascontiguousarray(coords), e.reshape(-1, 3)
    i = np.arange(n - 1, dtype=np.int32)
    v = ((i[:, None, None] * n + i[None, :, None]) * n + i[None, None, :]).ravel()
    step = (1, n, n * n)
    e = np.empty((v.size, 6, 4), np.int32)
    for q, p in enumerate(_PERMS):
        even = sum(p[x] > p[y] for x in range(3) for y in range(x + 1, 3)) % 2 == 0
        b, c = step[p[0]], step[p[0]] + step[p[1]]
        e[:, q, 0] = v
        e[:, q, 1] = v + (b if even else c)
        e[:, q, 2] = v + (c if even else b)
        e[:, q, 3] = v + 1 + n + n * n
    return np.ascontiguousarray(coords), e.reshape(-1, 4)


def _material(case, coords, elems, rng):
    """Young's modulus per element: one value, 1:100 on an 8 x 8 checkerboard of
    element centroids, or uniform in [1, 4]."""
    ne = elems.shape[0]
    if case["material"] == "checker":
        c = sum(coords[elems[:, q], :2] for q in range(elems.shape[1])) / elems.shape[1]
        odd = (np.floor(8.0 * c[:, 0]) + np.floor(8.0 * c[:, 1])).astype(np.int64) % 2
        E = np.where(odd == 0, 1.0, 100.0)
    elif case["material"] == "random":
        E = rng.uniform(1.0, 4.0, ne)
    else:
        E = np.full(ne, rng.uniform(1.0, 100.0))
    nu = case["nu"]
    return E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu)), E / (2.0 * (1.0 + nu))


def _measure(coords, elems):
    x0 = coords[elems[:, 0]]
    a = [coords[elems[:, q]] - x0 for q in range(1, elems.shape[1])]
    if len(a) == 2:
        return np.abs(a[0][:, 0] * a[1][:, 1] - a[0][:, 1] * a[1][:, 0]) / 2.0
    return np.abs(np.einsum("ij,ij->i", a[0], np.cross(a[1], a[2]))) / 6.0


def _problem(case, rng):
    """The problem dict of vasmg.Solver and its load vectors: each the
    consistent load of a constant body force of random direction, the x = 0
    edge / face clamped."""
    coords, elems = _mesh(case["dim"], case["n"], case["graded"], rng)
    d, nv = case["dim"], coords.shape[0]
    lam, mu = _material(case, coords, elems, rng)
    fixed = np.nonzero(coords[:, 0] == 0.0)[0].astype(np.int64)
    w = np.bincount(elems.ravel(), np.repeat(_measure(coords, elems) / (d + 1), d + 1), nv)
    F = [(w[:, None] * rng.uniform(-1.0, 1.0, d)[None, :]).ravel() for _ in range(case["k"] if case["kind"] == "multi" else 1)]
    return dict(dim=d, coords=coords, elems=elems, lam=lam, mu=mu,
                dirichlet_dofs=(fixed[:, None] * d + np.arange(d)[None, :]).ravel(), dirichlet_values=None), F


def _batch_case(case, i):
    """Mesh i of a batch: 2D of side n, 3D of side n/6, each a third smaller
    every other time; at least 24 and 9 vertices a side."""
    dim = 2 if i % 2 == 0 else 3
    n = case["n"] if dim == 2 else case["n"] // 6
    n = int(n * (2.0 / 3.0) ** (i // 2))
    return dict(case, kind="solve", dim=dim, n=max(24 if dim == 2 else 9, n), k=1)


def _problems(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "batch":
        return [_problem(_batch_case(case, i), rng) for i in range(case["k"])]
    return [_problem(case, rng)]


# ------------------------------------------------------------------ measured


def _solver(prob, precision, max_ctas=0):
    return vasmg.Solver(prob, precision=precision, stream=torch.cuda.current_stream().cuda_stream, max_ctas=max_ctas)


def prepare(case, seed):
    probs = _problems(case, seed)
    dev = [[torch.from_numpy(f).cuda() for f in F] for _, F in probs]
    st = dict(kind=case["kind"], precision=case["precision"], F=dev[0], U=[torch.zeros_like(f) for f in dev[0]])
    if case["kind"] == "request":
        st["prob"] = probs[0][0]
    elif case["kind"] == "batch":
        # the meshes share the device: each takes its part of the sweep grids
        st["solvers"] = [_solver(p, case["precision"], max_ctas=max(16, 128 // case["k"])) for p, _ in probs]
        st["F"] = [f[0] for f in dev]
        st["U"] = [torch.zeros_like(f) for f in st["F"]]
    else:
        st["solvers"] = [_solver(probs[0][0], case["precision"])]
        if case["kind"] == "update":
            p = probs[0][0]
            s = np.random.default_rng(seed + 1).uniform(0.5, 2.0, p["elems"].shape[0])
            st["prob"] = dict(p, lam=p["lam"] * s, mu=p["mu"] * s)
    return st


def run(st):
    kind = st["kind"]
    if kind == "request":
        s = _solver(st["prob"], st["precision"])
        rc = s.solve(st["F"][0], st["U"][0], TOL)[0]
        s.close()
    elif kind == "batch":
        rc = vasmg.vasmg_solve_batch([s.h for s in st["solvers"]], st["F"], st["U"], TOL)[0]
    elif kind == "multi":
        rc = st["solvers"][0].solve_multi(st["F"], st["U"], TOL)[0]
    else:
        if kind == "update":
            st["solvers"][0].update(st["prob"])
        rc = st["solvers"][0].solve(st["F"][0], st["U"][0], TOL)[0]
    return dict(status=rc, U=list(st["U"]))


# ------------------------------------------------------------------ needed work

# blocks per fine row (with the diagonal), operator blocks of all levels over
# the fine level's, and PCG iterations to 1e-8, for the meshes above
_ROW = {2: 7.0, 3: 15.0}
_SIZE = {"fp64": 8, "fp32": 4, "bf16": 2}


def _work1(c):
    d, nv = c["dim"], float(c["n"]) ** c["dim"]
    blocks = _ROW[d] * nv
    levels = 4.0 if d == 2 else (9.0 if c["graded"] != 1.0 else 5.0)
    iters = (16.0 if c["nu"] < 0.4 else 26.0) * (1.0 + (c["graded"] != 1.0)) * (4.0 if c["material"] == "checker" else 1.0)
    s = _SIZE[c["precision"]]
    # per iteration: the FP64 operator once; the V-cycle's operators twice (the
    # pre-smoothing's part, the residual's part, the post-smoothing's whole);
    # the vectors once in and once out
    nbytes = blocks * (8 * d * d + 4) + 2 * levels * blocks * (s * d * d + 4)
    flops = 2 * d * d * blocks * (1 + 2 * levels)
    vec = 8 * 10 * d * nv
    return iters * nbytes, iters * vec, iters * flops


def work(case):
    if case["kind"] == "batch":
        parts = [_work1(_batch_case(case, i)) for i in range(case["k"])]
        return {"bytes": sum(a + b for a, b, _ in parts), "flops": sum(f for _, _, f in parts)}
    a, b, f = _work1(case)
    return {"bytes": a + case["k"] * b, "flops": case["k"] * f}


# ------------------------------------------------------------------ in 64 bits


def _exact1(prob, F):
    """The solution for each load by block-Jacobi CG in 64 bits, the operator
    applied element by element; None where that takes too long."""
    d = prob["dim"]
    m = d + 1
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    X = torch.from_numpy(prob["coords"]).to(dev)
    E = torch.from_numpy(prob["elems"]).to(dev).long()
    lam, mu = (torch.from_numpy(np.broadcast_to(prob[q], (E.shape[0],)).copy()).to(dev) for q in ("lam", "mu"))
    n = X.shape[0] * d
    P = X[E]
    J = P[:, 1:] - P[:, :1]                       # rows: edges
    G = torch.linalg.inv(J).transpose(1, 2)       # gradients of the hats 1..d
    G = torch.cat([-G.sum(1, keepdim=True), G], 1)
    vol = torch.linalg.det(J).abs() / (2.0 if d == 2 else 6.0)
    gg = torch.einsum("eia,ejb->eiajb", G, G)
    I = torch.eye(d, dtype=torch.float64, device=dev)
    K = lam[:, None, None, None, None] * gg + mu[:, None, None, None, None] * (
        torch.einsum("eibja->eiajb", gg) + torch.einsum("eic,ejc,ab->eiajb", G, G, I))
    K = (K * vol[:, None, None, None, None]).reshape(-1, m * d, m * d)
    ids = (E[:, :, None] * d + torch.arange(d, device=dev)).reshape(-1, m * d)
    del gg, G, J, P
    free = torch.ones(n, dtype=torch.float64, device=dev)
    free[torch.from_numpy(np.asarray(prob["dirichlet_dofs"])).to(dev)] = 0.0
    D = torch.zeros(X.shape[0], d, d, dtype=torch.float64, device=dev)
    for q in range(m):
        D.index_add_(0, E[:, q], K[:, q * d:(q + 1) * d, q * d:(q + 1) * d])
    f2 = free.reshape(-1, d)
    D = D * f2[:, :, None] * f2[:, None, :] + torch.diag_embed(1.0 - f2)
    D = torch.linalg.inv(D)
    flat = ids.reshape(-1)

    def mul(x):
        y = torch.bmm(K, x[ids][:, :, None]).reshape(-1)
        return torch.zeros_like(x).index_add_(0, flat, y) * free

    most = 20000 if d == 2 else 3000
    out = []
    for f in F:
        r = torch.from_numpy(f).to(dev) * free
        x, p, rho, r0 = torch.zeros_like(r), None, None, float(r.norm())
        done = False
        for it in range(most):
            z = torch.bmm(D, r.reshape(-1, d, 1)).reshape(-1)
            rn = torch.dot(r, z)
            p = z if p is None else z + (rn / rho) * p
            rho = rn
            q = mul(p)
            a = rho / torch.dot(p, q)
            x = x + a * p
            r = r - a * q
            if it % 50 == 49 and float(r.norm()) <= 1e-13 * r0:
                done = True
                break
        out.append(x if done else None)
    return out


def exact(case, seed):
    probs = _problems(case, seed)
    elems = sum(p["elems"].shape[0] for p, _ in probs)
    if elems > (700_000 if case["dim"] == 2 else 1_600_000):
        return None
    if case["kind"] == "update":
        p = probs[0][0]
        s = np.random.default_rng(seed + 1).uniform(0.5, 2.0, p["elems"].shape[0])
        probs = [(dict(p, lam=p["lam"] * s, mu=p["mu"] * s), probs[0][1])]
    U = [u for p, F in probs for u in _exact1(p, F[:2])]
    if case["kind"] == "multi":
        U += [None] * (case["k"] - len(U))
    if all(u is None for u in U):
        return None
    return dict(status=None, U=U)
