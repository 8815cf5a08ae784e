"""Setup's sorts at the edges of their sizes.

Arrays of up to 4096 keys are sorted by one CTA, larger ones by tiles of 4096,
and pairs by the bits their words have.  So meshes whose vertex counts lie
around 256 (one digit more), around 4096 (the one-CTA sort's limit) and at the
smallest sizes build the same tree, transfer, pattern and colours as the
oracle, exactly.
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2505_09064_gb300 import meshgen, vasmg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n", [(2, 2), (2, 15), (2, 16), (2, 17), (2, 63), (2, 64), (2, 65), (2, 257),
                                   (3, 2), (3, 6), (3, 7), (3, 15), (3, 16), (3, 17)])
def test_setup_structure(dim, n):
    import __graft_entry__

    __graft_entry__.build()
    p = meshgen.make_problem(None, dim=dim, n=n, jitter=0.2 if dim == 2 else 0.15, seed=401)
    o = oracle.Oracle(p)
    s = vasmg.Solver(p, stream=torch.cuda.current_stream().cuda_stream)
    try:
        assert s.num_levels == o.num_levels
        assert np.array_equal(s.export(vasmg.EXPORT_MORTON, 0, np.uint64), o.morton())
        assert np.array_equal(s.export(vasmg.EXPORT_LEAF, 0, np.int64).reshape(-1, 2), o.leaves())
        for l in range(o.num_levels):
            assert np.array_equal(s.export(vasmg.EXPORT_A_CI, l, np.int32), o.operator(l)[1]), l
            assert np.array_equal(s.export(vasmg.EXPORT_COLOUR, l, np.int32), o.colours(l)), l
            if l + 1 < o.num_levels:
                assert np.array_equal(s.export(vasmg.EXPORT_P_CI, l, np.int32), o.prolongation(l)[1]), l
    finally:
        s.close()
