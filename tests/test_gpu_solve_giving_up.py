"""A solve whose thread blocks do not answer one another in time: the wait ends, the status says so and the result cannot pass
for a solution; the next solve in the same workspace is not affected.  (The wait is made to run out by allowing no polls.)"""
from __future__ import annotations

import ctypes

import pytest
import torch

from paper_2405_02508_gb300 import binding as B
from paper_2405_02508_gb300 import scenes
from paper_2405_02508_gb300.precond import LaplacianPreconditioner

pytestmark = pytest.mark.gpu


def _solve(pc, b, x, max_polls, launches=0):
    f = B.lib().mer_launch_precond_solve
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_float, ctypes.c_void_p, ctypes.c_void_p,
                  ctypes.c_int, ctypes.c_float, ctypes.c_void_p, ctypes.c_uint, ctypes.c_int, ctypes.c_void_p]
    return f(pc.row_ptr.data_ptr(), pc.col.data_ptr(), pc.V, pc.lam, b.data_ptr(), x.data_ptr(), pc.max_iters, pc.rel_tol,
             pc.workspace.data_ptr(), max_polls, launches, B._stream())


@pytest.mark.parametrize("n", [47, 64, 128])  # 8,838, 16,386 and 65,538 rows: several clusters, one and two rows a thread
def test_giving_up(n):
    P, F = scenes.octasphere(n)
    pc = LaplacianPreconditioner(F, len(P), 16.0)
    b = torch.randn((pc.V, 3), generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    want = pc.solve(b)
    x = torch.zeros_like(b)
    assert _solve(pc, b, x, 0) == B.MER_OK
    with pytest.raises(B.MerError) as e:
        pc.last_solve()
    assert e.value.code == B.MER_ECUDA
    assert torch.isnan(x).any()
    assert torch.equal(pc.solve(b), want) and pc.last_solve()[0] > 0


@pytest.mark.parametrize("n", [8, 32])  # one CTA and one cluster exchange nothing in memory: no poll to run out
def test_nothing_to_wait_for(n):
    P, F = scenes.octasphere(n)
    pc = LaplacianPreconditioner(F, len(P), 16.0)
    b = torch.randn((pc.V, 3), generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    x = torch.zeros_like(b)
    assert _solve(pc, b, x, 0) == B.MER_OK
    assert torch.equal(x, pc.solve(b))
