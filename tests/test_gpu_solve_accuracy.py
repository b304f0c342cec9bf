"""The one-launch preconditioner solve against the fixed launch sequence, whose dot products are FP64: the same number of
iterations to one, and the true residual of either (FP64, on meshes of bounded degree) within what FP32 vectors allow."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest
import torch

from paper_2405_02508_gb300 import binding as B
from paper_2405_02508_gb300 import scenes
from paper_2405_02508_gb300.precond import LaplacianPreconditioner

pytestmark = pytest.mark.gpu


def _launches(pc, b):
    f = B.lib().mer_launch_precond_solve
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_float, ctypes.c_void_p, ctypes.c_void_p,
                  ctypes.c_int, ctypes.c_float, ctypes.c_void_p, ctypes.c_uint, ctypes.c_int, ctypes.c_void_p]
    x = torch.zeros_like(b)
    assert f(pc.row_ptr.data_ptr(), pc.col.data_ptr(), pc.V, pc.lam, b.data_ptr(), x.data_ptr(), pc.max_iters, pc.rel_tol,
             pc.workspace.data_ptr(), 1 << 21, 1, B._stream()) == B.MER_OK
    return x


# 258, 902 rows: one CTA; 1,026 and 4,098: one cluster; then several, with one, two and four rows a thread
@pytest.mark.parametrize("n", [8, 15, 16, 32, 46, 64, 128, 181, 230])
@pytest.mark.parametrize("lam", [8.0, 32.0])
@pytest.mark.parametrize("smooth", [False, True])
def test_true_residual(n, lam, smooth):
    P, F = scenes.octasphere(n)
    pc = LaplacianPreconditioner(F, len(P), lam, max_iters=400)
    b = torch.randn((pc.V, 3), generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    if smooth:
        b = torch.from_numpy(P.astype(np.float32)).cuda() + 0.01 * b
    deg = pc.row_ptr.diff()
    rows, col = torch.repeat_interleave(torch.arange(pc.V, device="cuda"), deg), pc.col.long()
    its = []
    for solve in (pc.solve, lambda v: _launches(pc, v)):
        x = solve(b).double()
        it, _ = pc.last_solve()
        its.append(it)
        Mx = x + lam * (deg.double()[:, None] * x - torch.zeros_like(x).index_add_(0, rows, x[col]))
        # Each iteration rounds M p and the two updates of a row by at most 2^-24 (1 + 2 lam deg) of the row's and its
        # neighbours' values; over the iterations that adds up like a random walk.  The recursive residual is at most
        # rel_tol |b|.  (The same recurrence in FP32 on a CPU stays 5 to 8 times below.)
        big = torch.scatter_reduce(x.abs(), 0, rows[:, None].expand(-1, 3), x[col].abs(), "amax")
        rounding = 2.0 ** -24 * float(((1 + 2 * lam * deg.double())[:, None] * big).norm())
        assert float((b.double() - Mx).norm()) <= pc.rel_tol * float(b.double().norm()) + rounding * (it ** 0.5 + 1)
    assert 0 < its[0] < 400 and abs(its[0] - its[1]) <= 1
