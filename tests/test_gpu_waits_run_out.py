"""Every bounded device wait gives up, without a GPU fault.

The waits of the sweeps (a region's stage word, one tagged value, several
tagged values at once, a chunk of the staged operator) run in one CTA against
words that nothing writes: each must report VASMG_ERR_TIMEOUT after a bounded
time.  The tail's waits run out inside the tail itself, in a cluster whose last
CTA sends none of its rows: the other CTAs leave their sweeps, take part in no
further one, and the launch ends.  Afterwards the same hierarchy gives the same
bits as before.
"""
from __future__ import annotations

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


@pytest.mark.parametrize("which", [vasmg.WAIT_STAGE, vasmg.WAIT_TAGGED, vasmg.WAIT_TAGGED_ALL, vasmg.WAIT_CHUNK])
def test_wait_gives_up(built, which):
    rc, ms = vasmg.vasmg_probe_wait(which)
    assert rc == vasmg.VASMG_ERR_TIMEOUT
    assert 1.0 < ms < 10000.0


def test_unknown_wait_is_refused(built):
    assert vasmg.vasmg_probe_wait(4)[0] == vasmg.VASMG_ERR_INVALID_ARG
    assert vasmg.vasmg_probe_wait(-1)[0] == vasmg.VASMG_ERR_INVALID_ARG


@pytest.mark.parametrize("n", [33, 64, 220])
def test_tail_gives_up_and_recovers(built, n):
    prob = meshgen.make_problem(None, dim=2, n=n, jitter=0.2, seed=5)
    s = vasmg.Solver(prob, precision="fp32", stream=torch.cuda.current_stream().cuda_stream)
    try:
        F, U, V = (torch.zeros(s.n, dtype=torch.float64, device="cuda") for _ in range(3))
        s.assemble_load(prob["body_force"], F)
        assert s.solve(F, U, 1e-8)[0] == 0
        rc, ms = vasmg.vasmg_probe_tail_wait(s.h)
        assert rc == vasmg.VASMG_ERR_TIMEOUT
        assert 1.0 < ms < 20000.0
        assert s.solve(F, V, 1e-8)[0] == 0
        assert torch.equal(U, V)
    finally:
        s.close()
