"""Device memory of several right-hand sides' tagged values.

Sweeps of up to 4 right-hand sides wait for tagged values, 16 bytes per vertex
and right-hand side of every level with a staged copy; sweeps of 8 do not read
them.  So a handle that solved 8 right-hand sides holds twice the memory of
one that solved 4, less the words; the words come with its first pass of 4 or
fewer, and the results stay bitwise those of single solves whichever pass came
first.
"""
from __future__ import annotations

import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2505_09064_gb300 import meshgen, vasmg  # noqa: E402

pytestmark = pytest.mark.gpu

USED_MEM_CURRENT = 7  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT


@pytest.fixture(scope="module")
def built():
    import __graft_entry__

    __graft_entry__.build()
    torch.cuda.set_device(0)
    return True


def _used():
    """Bytes held from the device's stream-ordered pool, the library's allocator."""
    cu = C.CDLL("libcuda.so.1")
    pool, n = C.c_void_p(), C.c_uint64()
    torch.cuda.synchronize()
    assert cu.cuDeviceGetDefaultMemPool(C.byref(pool), C.c_int(torch.cuda.current_device())) == 0
    assert cu.cuMemPoolGetAttribute(pool, C.c_int(USED_MEM_CURRENT), C.byref(n)) == 0
    return n.value


def test_words_only_for_passes_that_read_them(built):
    prob = meshgen.make_problem(None, dim=3, n=41, jitter=0.15, seed=81)
    stream = torch.cuda.current_stream().cuda_stream
    four = vasmg.Solver(prob, precision="fp32", stream=stream)
    eight = vasmg.Solver(prob, precision="fp32", stream=stream)
    try:
        Fs, single = [], []
        for i in range(8):
            F, U = (torch.zeros(four.n, dtype=torch.float64, device="cuda") for _ in range(2))
            four.assemble_load(np.array([1.0, 0.5 * i, -0.25]), F)
            assert four.solve(F, U, 1e-6)[0] == 0
            Fs.append(F)
            single.append(U)
        lanes = four.export(vasmg.EXPORT_LANES, 0, np.int32)
        words = sum(four.level_info(l)[0] for l in range(four.num_levels) if lanes[l]) * 16

        def grows(s, k):
            Us = [torch.zeros_like(F) for F in Fs[:k]]
            before = _used()
            assert s.solve_multi(Fs[:k], Us, 1e-6)[0] == 0
            after = _used()
            for i in range(k):
                assert torch.equal(Us[i], single[i]), (k, i)
            return after - before

        m4 = grows(four, 4)
        m8 = grows(eight, 8)
        slack = 1 << 20  # per-pass constants and the pool's rounding of each array
        assert words * 8 > 4 * slack
        assert m8 <= 2 * m4 - 8 * words + slack, (m4, m8, words)
        assert abs(grows(eight, 3) - 4 * words) <= slack  # a pass of 4
        assert grows(eight, 2) <= 0
        assert grows(eight, 8) <= 0
        assert grows(four, 2) <= 0
    finally:
        four.close()
        eight.close()
