"""The raster's lane groups at their edges: triangles whose pixel boxes hold exactly the sizes at which a triangle moves to
a larger group (and one pixel less and more), long and flat ones among them, in both facings and overlapping, crossing the
bin tiles' borders, against the oracle's index image."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2405_02508_gb300.scenes import Shading

from . import parity
from .test_gpu_parity import gpu_screen_run, oracle_screen_run

pytestmark = pytest.mark.gpu

# (width, height) in pixel centres: 1, 2, 7, 8, 9, 63, 64, 65 pixels and boxes wider or taller than any tile
BOXES = [(1, 1), (2, 1), (1, 2), (7, 1), (2, 4), (8, 1), (1, 8), (3, 3), (9, 7), (7, 9), (8, 8), (64, 1), (1, 64), (5, 13),
         (13, 5), (16, 16), (17, 15), (70, 2), (2, 70), (70, 70)]


@pytest.fixture(scope="module")
def orc():
    import oracle

    oracle.build()
    return oracle


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("per_box", [1, 40])
def test_box_sizes(orc, tile, per_box):
    H, W = 97, 131
    rng = np.random.default_rng(per_box)
    pts = []
    for w, h in BOXES:
        for k in range(per_box):
            x, y = rng.integers(-4, W - 2), rng.integers(-4, H - 2)
            # corners just outside the first and last centre of the box: every centre on its border stays inside it
            lo, hi = np.array([x + 0.45, y + 0.45]), np.array([x + w - 0.45, y + h - 0.45])
            third = rng.uniform(lo, hi)
            tri = [[lo[0], lo[1]], [hi[0], lo[1]], [third[0], hi[1]]]
            if k % 2 == 0:
                tri = tri[::-1]
            pts.append(np.concatenate([np.array(tri), rng.uniform(0.2, 1.0, (3, 1))], axis=1))
    scr = np.concatenate(pts)
    nt = len(pts)
    tris = np.arange(3 * nt, dtype=np.int32).reshape(nt, 3)
    sh = Shading(n_main=1, C=1, bg=[0.25])
    attr = rng.uniform(0.1, 0.9, (3 * nt, 1)).astype(np.float32)
    g = rng.standard_normal((1, H, W, 1)).astype(np.float32)
    gi, gimg, _ = gpu_screen_run(scr, tris, H, W, sh, attr, g, tile=tile)
    oi, tie, oimg, _, _ = oracle_screen_run(orc, scr, tris, H, W, sh, attr, g[0])
    assert np.all((gi == oi) | tie)
    same = gi == oi
    np.testing.assert_allclose(gimg[same], oimg[same], rtol=parity.IMG_TOL, atol=parity.IMG_TOL)
