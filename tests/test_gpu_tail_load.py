"""The tail's clusters beside other work on the device.

The CTAs of a tail cluster exchange the rows of a colour through each other's
shared memory.  Alone on the device they keep step; with other kernels on some
of their SMs one of them can lag another by far more than a colour step, and
whatever order the values rely on has to come from barriers.  So a hierarchy
solves again and again while another handle of the same problem solves on a
second stream and small kernels fill the device from a third, and every result
is bitwise the one of a solve with the device to itself (no order of additions
depends on the CTAs' progress).
"""
from __future__ import annotations

import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2505_09064_gb300 import meshgen, vasmg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def built():
    import __graft_entry__

    __graft_entry__.build()
    torch.cuda.set_device(0)
    return True


class _Load(threading.Thread):
    """A second handle's solves and a stream of small kernels, until stopped."""

    def __init__(self, prob, precision):
        super().__init__(daemon=True)
        self.stop = threading.Event()
        self.error = None
        self.stream, self.fill = torch.cuda.Stream(), torch.cuda.Stream()
        self.s = vasmg.Solver(prob, precision=precision, stream=self.stream.cuda_stream, max_ctas=64)
        self.a = torch.ones(1 << 22, device="cuda")
        self.solves = 0

    def run(self):
        try:
            torch.cuda.set_device(0)
            F, U = (torch.zeros(self.s.n, dtype=torch.float64, device="cuda") for _ in range(2))
            torch.cuda.synchronize()
            self.s.assemble_load(np.full(self.s.dim, 0.5), F)
            while not self.stop.is_set():
                with torch.cuda.stream(self.fill):
                    for _ in range(200):
                        self.a.mul_(1.0)
                rc, _, _ = self.s.solve(F, U, 1e-8)
                assert rc == 0
                self.fill.synchronize()
                self.solves += 1
        except Exception as e:  # noqa: BLE001  (reported by the test)
            self.error = e


def _solve_under_load(dim, n, precision, repeats=100):
    prob = meshgen.make_problem(None, dim=dim, n=n, jitter=0.2 if dim == 2 else 0.15, seed=501, nu=0.35)
    stream = torch.cuda.Stream()
    s = vasmg.Solver(prob, precision=precision, stream=stream.cuda_stream, max_ctas=64)
    load = _Load(prob, precision)
    try:
        F, alone, U = (torch.zeros(s.n, dtype=torch.float64, device="cuda") for _ in range(3))
        torch.cuda.synchronize()
        s.assemble_load(prob["body_force"], F)
        rc, st, _ = s.solve(F, alone, 1e-8)
        assert rc == 0
        torch.cuda.synchronize()
        load.start()
        for k in range(repeats):
            rc, sk, _ = s.solve(F, U, 1e-8)
            assert rc == 0 and sk.iterations == st.iterations, k
            stream.synchronize()
            assert torch.equal(U, alone), (k, float((U - alone).abs().max()))
    finally:
        load.stop.set()
        if load.ident is not None:
            load.join(60)
        s.close()
        load.s.close()
    assert load.error is None, load.error
    assert load.solves > 0


@pytest.mark.parametrize("dim,n,precision", [(2, 64, "fp64"), (3, 17, "fp32")])
def test_copies_filled_before_rows_arrive(built, dim, n, precision):
    """Every level of these tails has its x in every CTA's shared memory, filled
    from global memory before each backward sweep sends its rows into it."""
    _solve_under_load(dim, n, precision)


@pytest.mark.parametrize("dim,n,precision", [(3, 24, "fp32"), (3, 17, "fp64"), (2, 141, "fp64"), (2, 220, "fp32")])
def test_level_below_in_the_copies(built, dim, n, precision):
    """A level of these tails does not fit the CTAs' shared memory and the next
    coarser one does: the prolongation reads values that other CTAs wrote to
    global memory during the coarser level's sweep."""
    _solve_under_load(dim, n, precision)
