"""The operator tests hold coarse rows of both kinds.

A coarse row's Galerkin sum goes through a table of at most 192 (2D) or 768
(3D) fine columns, and rows that reach more of them are summed by another
kernel; the operators do not tell which ran.  So the meshes of
test_gpu_galerkin.py and test_gpu_galerkin_wide.py are counted here: the distinct
fine columns of the fine rows that a coarse row restricts, from the oracle's P
and A.  Rows stay within the table in the former (in 2D some exceed it), and
every case of the latter has rows beyond it, in 2D and in 3D.
"""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import test_gpu_galerkin
import test_gpu_galerkin_wide
from paper_2505_09064_gb300 import meshgen

TABLE = {2: 192, 3: 768}  # three quarters of the slots of setup_galerkin.cu


def _reach(o, l):
    """Distinct fine columns per coarse row of level l + 1."""
    arp, aci, _ = o.operator(l)
    prp, pci, _ = o.prolongation(l)
    rows = [[] for _ in range(o.nv_level(l + 1))]
    for i in range(o.nv_level(l)):
        for J in pci[prp[i]:prp[i + 1]]:
            rows[J].append(aci[arp[i]:arp[i + 1]])
    return np.array([np.unique(np.concatenate(r)).size if r else 0 for r in rows])


def _cases():
    mark = next(m for m in test_gpu_galerkin.test_coarse_operators.pytestmark if m.name == "parametrize")
    return mark.args[1]


def _count(o, dim):
    r = [_reach(o, l) for l in range(o.num_levels - 1)]
    return sum(int((a > TABLE[dim]).sum()) for a in r), sum(int((a <= TABLE[dim]).sum()) for a in r)


@pytest.mark.parametrize("dim", [2, 3])
def test_rows_within_the_table(dim):
    narrow = 0
    for d, n, threshold in _cases():
        if d == dim:
            p = meshgen.make_problem(None, dim=d, n=n, jitter=0.2 if d == 2 else 0.15, seed=301, nu=0.4)
            narrow += _count(oracle.Oracle(p, threshold=threshold), d)[1]
    assert narrow > 0


@pytest.mark.parametrize("name", list(test_gpu_galerkin_wide.CASES))
def test_rows_beyond_the_table(name):
    make, threshold = test_gpu_galerkin_wide.CASES[name]
    p = make()
    o = oracle.Oracle(p, threshold=threshold) if threshold else oracle.Oracle(p)
    wide, _ = _count(o, p["dim"])
    assert wide > 0
    if name.startswith("disc"):
        assert np.diff(o.operator(0)[0]).max() > 1023
