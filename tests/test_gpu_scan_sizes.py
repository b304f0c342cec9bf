"""Binning at tile counts around the edges of the scan: one count, a row of a warp, a thread's first and last row, and the first
size that takes several launches.  The bins decide the index image, which does not depend on the tile size."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2405_02508_gb300 import binding as B
from paper_2405_02508_gb300 import scenes

pytestmark = pytest.mark.gpu


# views and tiles of 8 x 8 down and across: 1, 31, 33, 1,023 to 1,025, 2,047, 2,049, 4,097 and 15,376 to 16,385 counts
@pytest.mark.parametrize("views,ny,nx", [(1, 1, 1), (31, 1, 1), (3, 1, 11), (1, 31, 33), (1, 32, 32), (1, 25, 41), (1, 23, 89),
                                         (1, 3, 683), (17, 1, 241), (1, 124, 124), (1, 129, 127), (1, 128, 128), (5, 29, 113)])
def test_index_at_scan_sizes(views, ny, nx):
    H, W = 8 * ny - 3, 8 * nx - 3
    P, F = scenes.octasphere(20)
    verts = torch.from_numpy(P.astype(np.float32)).cuda()
    tris = torch.from_numpy(F.astype(np.int32)).cuda()
    vpix = torch.zeros((views, len(P), B.VERTEX_FLOATS), device="cuda")
    B.mer_project(verts, B.cameras_tensor(scenes.cameras_on_sphere(views, 3.0, H, W, 2)), vpix)
    out = {}
    for tile in (8, 32):
        index = torch.full((views, H, W), -9, dtype=torch.int32, device="cuda")
        capacity = 0
        for _ in range(3):  # the first time to size the lists, the third over what the second left in the workspace
            if capacity >= 0:
                ws = torch.zeros(B.mer_workspace_size(len(P), len(F), views, H, W, tile, capacity) // 4, device="cuda")
            B.mer_rasterize(vpix, tris, H, W, tile, ws, index)
            code, total = B.mer_sync_status(ws)
            capacity = total if capacity == 0 else -1
        assert code == B.MER_OK and total > 0
        out[tile] = index
    assert (out[8] >= 0).any() and torch.equal(out[8], out[32])
