"""Preconditioner solves with rows of many neighbours, on both sides of the number up to which a thread sums its own row, one or
several in a warp, in every form of the solve: the true residual (FP64) stays within what FP32 vectors allow, row by row."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2405_02508_gb300.precond import LaplacianPreconditioner

pytestmark = pytest.mark.gpu


def _mesh(V: int, hubs: list[int]) -> np.ndarray:
    """A strip over V vertices, and a fan of d triangles around vertex 3 h for the h-th number d: d + 1 neighbours or a few more."""
    i = np.arange(V - 2)
    tris = [np.stack([i, i + 1, i + 2], 1)]
    rng = np.random.default_rng(V)
    for h, d in enumerate(hubs):
        ring = rng.permutation(np.arange(3 * len(hubs), V))[: d + 1]
        tris.append(np.stack([np.full(d, 3 * h), ring[:-1], ring[1:]], 1))
    return np.concatenate(tris).astype(np.int32)


@pytest.mark.parametrize("V", [1000, 3000, 8000, 20000, 65538, 140001])
@pytest.mark.parametrize("hubs", [[56], [59, 60, 61, 62, 63], [64], [100] * 12, [300, 20, 900]])
def test_rows_of_many_neighbours(V, hubs):
    lam = 16.0
    pc = LaplacianPreconditioner(_mesh(V, hubs), V, lam, max_iters=400)
    b = torch.randn((V, 3), generator=torch.Generator(device="cuda").manual_seed(V), device="cuda")
    x = pc.solve(b).double()
    it, res = pc.last_solve()
    assert 0 < it < 400 and res <= pc.rel_tol
    deg = pc.row_ptr.diff()
    rows, col = torch.repeat_interleave(torch.arange(V, device="cuda"), deg), pc.col.long()
    Mx = x + lam * (deg.double()[:, None] * x - torch.zeros_like(x).index_add_(0, rows, x[col]))
    # as for meshes of bounded degree: 2^-24 (1 + 2 lam deg) of the largest value of the row and its neighbours an
    # iteration, adding up like a random walk
    big = torch.scatter_reduce(x.abs(), 0, rows[:, None].expand(-1, 3), x[col].abs(), "amax")
    rounding = 2.0 ** -24 * float(((1 + 2 * lam * deg.double())[:, None] * big).norm())
    assert float((b.double() - Mx).norm()) <= pc.rel_tol * float(b.double().norm()) + rounding * (it ** 0.5 + 1)
