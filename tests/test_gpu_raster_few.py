"""Tiles with few triangles, on both sides of the number up to which a warp takes each: the index image does not depend on the
tile size, with overlapping triangles of small and full boxes, front and back facing, equal depths among them."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2405_02508_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_tile", [1, 2, 7, 8, 9, 10, 31, 33])
def test_few_triangles(per_tile):
    H, W = 45, 61
    rng = np.random.default_rng(per_tile)
    tri = []
    for ty in range(0, H, 16):
        for tx in range(0, W, 16):
            for k in range(per_tile):
                size = (3.0, 6.0, 15.5)[k % 3]
                c = np.array([tx, ty]) + rng.uniform(0, 16 - size if size < 16 else 0.4, 2)
                p = c + rng.uniform(0, size, (3, 2))
                z = rng.uniform(0.2, 0.6, (3, 1)) if k % 4 else np.full((3, 1), 0.5)
                tri.append(np.concatenate([p, z], 1))
    scr = torch.from_numpy(np.stack(tri).reshape(1, -1, 3)).cuda()
    tris = torch.arange(scr.shape[1], dtype=torch.int32, device="cuda").view(-1, 3)
    vpix = torch.zeros((1, scr.shape[1], B.VERTEX_FLOATS), device="cuda")
    B.mer_project_screen(scr, vpix)
    out = []
    for tile in (32, 16, 8):
        ws = torch.zeros(B.mer_workspace_size(scr.shape[1], len(tris), 1, H, W, tile, 64 * len(tris)) // 4, device="cuda")
        index = torch.full((1, H, W), -9, dtype=torch.int32, device="cuda")
        cover = torch.zeros((1, H, W), dtype=torch.uint8, device="cuda")
        B.mer_rasterize(vpix, tris, H, W, tile, ws, index, cover=cover)
        assert B.mer_sync_status(ws)[0] == B.MER_OK
        out.append((index, cover & B_WINNER))
    assert (out[0][0] >= 0).any()
    for index, winner in out[1:]:
        assert torch.equal(index, out[0][0]) and torch.equal(winner, out[0][1])


B_WINNER = 4  # MER_COVER_WINNER_BACK: the other bits of the cover image depend on the tile's border
