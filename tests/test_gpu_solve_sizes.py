"""The preconditioner's solve at the edges of its forms: one CTA, one cluster, several clusters, one, two and four rows a
thread, and sizes beyond one resident grid, against conjugate gradients in FP64 (plain torch) of the same system."""
from __future__ import annotations

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _strip(V: int) -> np.ndarray:
    """A triangulated strip over V vertices in shuffled order, plus a fan of 40 triangles around vertex 0 (a row with
    more neighbours than a thread keeps in registers); the last vertex of an odd tail may stay isolated."""
    perm = np.random.default_rng(V).permutation(V)
    i = np.arange(V - 3)
    tris = np.stack([i, i + 1, i + 2], 1)  # vertex V - 1 is isolated
    fan = np.stack([np.zeros(40, np.int64), 1 + np.arange(40) % (V - 2), 1 + (np.arange(40) + 1) % (V - 2)], 1)
    return perm[np.concatenate([tris, fan])].astype(np.int32)


def _solve64(row_ptr, col, lam, b):
    rows = torch.repeat_interleave(torch.arange(len(row_ptr) - 1, device="cuda"), row_ptr.diff())
    deg = row_ptr.diff().double()[:, None]
    col = col.long()

    def M(x):
        return x + lam * (deg * x - torch.zeros_like(x).index_add_(0, rows, x[col]))

    b = b.double()
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), (r * r).sum()
    stop = 1e-26 * rr
    for _ in range(2000):
        if rr <= stop:
            break
        q = M(p)
        a = rr / (p * q).sum()
        x, r = x + a * p, r - a * q
        new = (r * r).sum()
        p, rr = r + (new / rr) * p, new
    return x, M


@pytest.mark.parametrize("V", [5, 31, 1023, 1024, 1025, 4095, 4096, 4097, 8192, 8193, 32769, 65538, 140001, 270001])
@pytest.mark.parametrize("scale", [1.0, 1e-21, 1e18])
def test_solve_at_form_edges(V, scale):
    from paper_2405_02508_gb300.precond import LaplacianPreconditioner

    if scale != 1.0 and V > 9000:
        pytest.skip("scales at the small forms")
    lam, tol = 16.0, 1e-6
    pc = LaplacianPreconditioner(_strip(max(V, 5)), V, lam, max_iters=400, rel_tol=tol)
    b = scale * torch.randn((V, 3), generator=torch.Generator(device="cuda").manual_seed(V), device="cuda")
    x = pc.solve(b)
    it, res = pc.last_solve()
    ref, M = _solve64(pc.row_ptr, pc.col[: int(pc.row_ptr[-1])], lam, b)
    assert 0 < it < 400 and res <= tol
    # the recursive residual is at most tol |b|; the true one adds FP32 rounding of each iteration's M p and updates,
    # at most 2^-24 (1 + 2 lam deg) |x| each, adding up like a random walk over the iterations
    deg = float(pc.row_ptr.diff().max())
    nb, nx = float((b.double() / scale).norm()), float((ref / scale).norm())
    bound = tol * nb + 2.0 ** -24 * (1 + 2 * lam * deg) * nx * (it ** 0.5 + 1)
    assert float(((M(x.double()) - b.double()) / scale).norm()) <= bound
    # all eigenvalues of M are at least 1
    assert float(((x.double() - ref) / scale).norm()) <= bound


def test_solve_under_capture_and_limits():
    """A captured solve replays to the same bits; the iteration limit and a zero right-hand side are kept."""
    from paper_2405_02508_gb300 import binding as B
    from paper_2405_02508_gb300.precond import LaplacianPreconditioner

    for V in (700, 3000, 20000):
        pc = LaplacianPreconditioner(_strip(V), V, 16.0)
        b = torch.randn((V, 3), generator=torch.Generator(device="cuda").manual_seed(V), device="cuda")
        x = pc.solve(b)
        out = torch.zeros_like(b)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            out.zero_()
            B.mer_precond_solve(pc.row_ptr, pc.col, pc.lam, b, out, pc.max_iters, pc.rel_tol, pc.workspace)
        for _ in range(2):
            g.replay()
            assert torch.equal(out, x)
        pc.max_iters = 3
        pc.solve(b)
        assert pc.last_solve()[0] == 3
        z = torch.zeros_like(b)
        assert torch.equal(pc.solve(z), z) and pc.last_solve()[0] == 0


def test_solves_on_two_streams():
    """Solves of different sizes on two streams at once, each in its own workspace."""
    from paper_2405_02508_gb300.precond import LaplacianPreconditioner

    pcs, bs, alone = [], [], []
    for V in (900, 6000, 40000, 65538):
        pc = LaplacianPreconditioner(_strip(V), V, 8.0)
        b = torch.randn((V, 3), generator=torch.Generator(device="cuda").manual_seed(V), device="cuda")
        pcs.append(pc)
        bs.append(b)
        alone.append(pc.solve(b))
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = []
    for k, (pc, b) in enumerate(zip(pcs, bs)):
        with torch.cuda.stream(streams[k % 2]):
            outs.append(pc.solve(b))
    torch.cuda.synchronize()
    for x, y in zip(outs, alone):
        assert torch.equal(x, y)
