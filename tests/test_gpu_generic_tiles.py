"""The generic layout at 64 x 64 tiles on both sides of the tile count from which it takes the variant with fewer registers (four
tiles a multiprocessor): both draw what the 16 x 16 tiles draw, bit for bit, whatever grid is asked for."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2405_02508_gb300 import scenes
from paper_2405_02508_gb300.batch import BatchRenderer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("over", [-1, 0, 1])
@pytest.mark.parametrize("ctas", [0, 1, 700, 5000])
def test_generic_at_64(over, ctas):
    tiles = 4 * torch.cuda.get_device_properties(0).multi_processor_count + over  # one item a tile
    P, F = scenes.octasphere(6)
    sh = scenes.Shading(n_main=2, C=4, mask_ch=3, backface_ch=2, bg=[0.2, 0.1, 0.0, 0.0])
    cams = scenes.cameras_on_sphere(8, 3.0, 61, 64, 2)
    attr = torch.from_numpy(np.random.default_rng(1).uniform(0, 1, (len(P), 2)).astype(np.float32)).cuda()
    verts = torch.from_numpy(P.astype(np.float32)).cuda()
    out = []
    for tile, grid in ((16, 0), (64, ctas)):
        br = BatchRenderer([(P, F.astype(np.int32))], [(0, k % 8, 61, 64) for k in range(tiles)], cams, sh, 2, None, tile=tile,
                           persistent_ctas=grid)
        br.prepare(verts, attr)
        assert tile != 64 or br.tot.tiles == tiles
        out.append((br.index, br.image))
    assert (out[0][0] >= 0).any()
    assert torch.equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1].view(torch.int32), out[1][1].view(torch.int32))
