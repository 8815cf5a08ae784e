"""Coarse rows that reach more fine columns than the Galerkin product's table takes.

Two kinds of meshes have them.  With a large leaf threshold a coarse cell holds
many fine vertices.  And a vertex may have many neighbours: a disc of four rings
of 1100 vertices around one centre, whose row holds 1101 blocks, also more than
the 1023 that a row length may have in the SpMV's sort key; all dofs of the rim
are fixed, and, in a second case, one component everywhere (its coarse dofs are
then dead in every row).

The structure and the operators of every level are the oracle's, an update of the
material gives bitwise the operators of a fresh setup, and the disc's solution is
the oracle's.
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2505_09064_gb300 import meshgen, vasmg  # noqa: E402

pytestmark = pytest.mark.gpu

RIM, RINGS = 1100, 4


def fan(fix_y):
    t = 2.0 * np.pi * np.arange(RIM) / RIM
    X = [np.zeros((1, 2))] + [r * np.stack([np.cos(t), np.sin(t)], 1) for r in range(1, RINGS + 1)]
    X = np.concatenate(X) / (2.0 * RINGS) + 0.5
    i, ip = np.arange(RIM), (np.arange(RIM) + 1) % RIM
    E = [np.stack([np.zeros(RIM, np.int64), 1 + i, 1 + ip], 1)]
    for r in range(1, RINGS):
        a, b = 1 + (r - 1) * RIM, 1 + r * RIM
        E += [np.stack([a + i, b + i, b + ip], 1), np.stack([a + i, b + ip, a + ip], 1)]
    E = np.concatenate(E).astype(np.int32)
    rim = np.arange(1 + (RINGS - 1) * RIM, 1 + RINGS * RIM)
    fixed = (rim[:, None] * 2 + np.arange(2)).ravel()
    if fix_y:
        fixed = np.unique(np.concatenate([fixed, 2 * np.arange(X.shape[0]) + 1]))
    rng = np.random.default_rng(7)
    mu = rng.uniform(1.0, 3.0, len(E))
    return dict(dim=2, coords=X, elems=E, lam=1.5 * mu, mu=mu, dirichlet_dofs=fixed.astype(np.int64),
                dirichlet_values=None, body_force=np.array([0.5, -1.0]))


def grid(dim, n):
    return meshgen.make_problem(None, dim=dim, n=n, jitter=0.2 if dim == 2 else 0.15, seed=301, nu=0.4)


# (problem, leaf threshold; 0: the default)
CASES = {
    "2d_40_200": (lambda: grid(2, 40), 200),
    "3d_14_1000": (lambda: grid(3, 14), 1000),
    "3d_17_100": (lambda: grid(3, 17), 100),
    "3d_20_300": (lambda: grid(3, 20), 300),
    "disc": (lambda: fan(False), 0),
    "disc_y_fixed": (lambda: fan(True), 0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_operators(name):
    import __graft_entry__

    __graft_entry__.build()
    make, threshold = CASES[name]
    p = make()
    d = p["dim"]
    q = dict(p, lam=p["lam"] * 3.0, mu=p["mu"] * 0.5)
    o = oracle.Oracle(q, threshold=threshold) if threshold else oracle.Oracle(q)
    stream = torch.cuda.current_stream().cuda_stream
    fresh = vasmg.Solver(q, stream=stream, threshold=threshold)
    upd = vasmg.Solver(p, stream=stream, threshold=threshold)
    try:
        upd.update(q)
        assert fresh.num_levels == o.num_levels
        top = 0.0
        for l in range(o.num_levels):
            _, oci, ov = o.operator(l)
            assert np.array_equal(fresh.export(vasmg.EXPORT_A_CI, l, np.int32), oci)
            v = fresh.export(vasmg.EXPORT_A_V, l, np.float64).reshape(-1, d, d)
            # a scalar of a coarse block sums at most the 28,601 blocks of the disc
            # (or 8 cells of 1000 vertices with 15 blocks each), each times two weights
            # of at most 1, every product and sum rounded to 2^-53 and most of them
            # far below the largest entry so far: 1e-11 of it
            top = max(top, float(np.abs(ov).max()))
            assert np.abs(v - ov).max() <= 1e-11 * top, l
            assert np.array_equal(v, upd.export(vasmg.EXPORT_A_V, l, np.float64).reshape(-1, d, d))
            assert np.array_equal(fresh.export(vasmg.EXPORT_DEAD, l, np.uint8), o.dead(l))
    finally:
        fresh.close()
        upd.close()


def test_disc_solution():
    import __graft_entry__

    __graft_entry__.build()
    p = fan(False)
    o = oracle.Oracle(p)
    F = o.assemble_load(p["body_force"])
    ref, iters, _, status, _ = o.solve(F, tol=1e-10)
    assert status == 0
    s = vasmg.Solver(p, stream=torch.cuda.current_stream().cuda_stream)
    try:
        Fd = torch.from_numpy(F).cuda()
        U = torch.zeros_like(Fd)
        rc, st, _ = s.solve(Fd, U, 1e-10)
        assert rc == 0 and abs(st.iterations - iters) <= 1
        assert np.linalg.norm(U.cpu().numpy() - ref) <= 1e-7 * np.linalg.norm(ref)
    finally:
        s.close()
