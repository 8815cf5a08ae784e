"""The Galerkin product's two ways of summing a coarse row.

A coarse row is summed through a table of the fine columns it reaches (up to
192 in 2D and 768 in 3D), or, when it reaches more of them, term by term.
With a large leaf threshold a coarse cell holds many fine vertices, so both
ways run here: the operators of every level equal the oracle's to 1e-12 of the
largest entry (a sum of at most a few thousand products of magnitude at most
that entry, each rounded to 2^-53, stays below 1e-12 of it), and an update of
the material gives bitwise the operators of a fresh setup.
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2505_09064_gb300 import meshgen, vasmg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,threshold", [(2, 3, 4), (2, 40, 4), (2, 40, 64), (2, 40, 200), (3, 3, 8), (3, 11, 8),
                                             (3, 14, 64), (3, 14, 300)])
def test_coarse_operators(dim, n, threshold):
    import __graft_entry__

    __graft_entry__.build()
    p = meshgen.make_problem(None, dim=dim, n=n, jitter=0.2 if dim == 2 else 0.15, seed=301, nu=0.4)
    q = dict(p, lam=p["lam"] * 3.0, mu=p["mu"] * 0.5)
    o = oracle.Oracle(q, threshold=threshold)
    stream = torch.cuda.current_stream().cuda_stream
    fresh = vasmg.Solver(q, stream=stream, threshold=threshold)
    upd = vasmg.Solver(p, stream=stream, threshold=threshold)
    try:
        upd.update(q)
        assert fresh.num_levels == o.num_levels
        for l in range(o.num_levels):
            orp, oci, ov = o.operator(l)
            assert np.array_equal(fresh.export(vasmg.EXPORT_A_CI, l, np.int32), oci)
            v = fresh.export(vasmg.EXPORT_A_V, l, np.float64).reshape(-1, dim, dim)
            assert np.abs(v - ov).max() <= 1e-12 * np.abs(ov).max(), l
            assert np.array_equal(v, upd.export(vasmg.EXPORT_A_V, l, np.float64).reshape(-1, dim, dim))
            assert np.array_equal(fresh.export(vasmg.EXPORT_DEAD, l, np.uint8), o.dead(l))
    finally:
        fresh.close()
        upd.close()
