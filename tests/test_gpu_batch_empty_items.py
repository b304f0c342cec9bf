"""Items without vertices in the batched projection backward: their camera index, which nothing uses, is not looked up."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2405_02508_gb300 import binding as B
from paper_2405_02508_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [1, 31, 32, 33, 255, 257])
def test_empty_items(V):
    cams = B.cameras_tensor(scenes.cameras_on_sphere(2, 3.0, 40, 40, 1))
    verts = torch.from_numpy(np.random.default_rng(V).normal(0, 0.3, (V, 3)).astype(np.float32)).cuda()
    grad = torch.randn((2 * V, 3), generator=torch.Generator(device="cuda").manual_seed(V), device="cuda").double()
    out = {}
    for empty in (False, True):
        sizes = [(0, 1 << 30), (V, 0), (0, 1 << 30), (V, 1), (0, 1 << 30)] if empty else [(V, 0), (V, 1)]
        arr = (B.MerItem * len(sizes))()
        for k, (v, cam) in enumerate(sizes):
            arr[k].V, arr[k].cam = v, cam
        tot = B.mer_batch_plan(arr, 32)
        items = torch.from_numpy(np.frombuffer(bytes(arr), dtype=np.uint8).copy()).cuda()
        vpix = torch.zeros((2 * V, B.VERTEX_FLOATS), device="cuda")
        gv = torch.zeros((V, 3), device="cuda")
        B.mer_batch_project(verts, cams, items, tot, vpix)
        B.mer_batch_project_backward(cams, items, tot, vpix, grad, gv)
        out[empty] = gv
    # two terms added to zero, in either order
    assert torch.equal(out[False], out[True]) and (out[True] != 0).any()
