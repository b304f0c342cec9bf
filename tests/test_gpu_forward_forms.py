"""The layout forms of the forward gradients against the generic form: a scene in a layout that only the generic form takes has
the same derivative image, in particular at texel borders, where a weight rounded otherwise reads another texel."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2405_02508_gb300 import binding as B
from paper_2405_02508_gb300 import scenes
from paper_2405_02508_gb300.render import Renderer

pytestmark = pytest.mark.gpu


def _derivative(sh, P, F, attr, tex, H, W, terms):
    r = Renderer(torch.from_numpy(F.astype(np.int32)), len(P), 2, H, W, sh, attr.shape[1], None if tex is None else tex.shape)
    verts, a = torch.from_numpy(P.astype(np.float32)).cuda(), torch.from_numpy(attr).cuda()
    t = None if tex is None else torch.from_numpy(tex).cuda()
    cams = B.cameras_tensor(scenes.cameras_on_sphere(2, 3.0, H, W, 3))
    r.forward(verts, cams, a, t)
    tangent = torch.randn(verts.shape, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda")
    return r.forward_grad(tangent, cams, a, t, terms=terms).cpu().numpy()


def _same(x, y):
    """A texel read instead of its neighbour changes a derivative by its own size; the roundings of a hundred operations are
    below 2^-17 of the largest."""
    for c in range(x.shape[-1]):
        np.testing.assert_allclose(x[..., c], y[..., c], rtol=0, atol=1e-3 * max(np.abs(y[..., c]).max(), 1e-30))


# about a pixel a triangle, a few, and many; coarse and fine texels; the vertices on texel borders
@pytest.mark.parametrize("n,H,W", [(110, 240, 260), (30, 301, 333), (4, 200, 150)])
@pytest.mark.parametrize("size", [(3, 5), (64, 64), (512, 512)])
@pytest.mark.parametrize("terms", [2, 7])
def test_textured(n, H, W, size, terms):
    P, F = scenes.octasphere(n)
    rng = np.random.default_rng(5)
    th, tw = size
    uv = scenes.equirect_uv(P).astype(np.float32)
    uv[::3] = (np.round(uv[::3] * [tw, th] - 0.5) + 0.5) / np.float32([tw, th])
    uv = uv.astype(np.float32)
    tex = rng.uniform(0, 1, (*size, 4)).astype(np.float32)
    sh = scenes.Shading(n_main=3, C=5, uv_offset=0, mask_ch=3, depth_ch=4, bg=[0.1, 0.2, 0.3, 0.0, 0.0])
    wide = np.concatenate([uv, rng.uniform(0, 1, (len(uv), 1)).astype(np.float32)], axis=1)  # three floats a vertex: generic
    _same(_derivative(sh, P, F, uv, tex, H, W, terms), _derivative(sh, P, F, wide, tex, H, W, terms))


@pytest.mark.parametrize("terms", [2, 7])
def test_interpolated(terms):
    P, F = scenes.octasphere(30)
    attr = np.random.default_rng(6).uniform(-1, 1, (len(P), 4)).astype(np.float32)
    four = scenes.Shading(n_main=4, C=5, mask_ch=4, bg=[0.1, 0.2, 0.3, 0.4, 0.0])  # four channels: generic
    three = scenes.Shading(n_main=3, C=4, mask_ch=3, bg=[0.1, 0.2, 0.3, 0.0])
    y = _derivative(four, P, F, attr, None, 301, 333, terms)
    x = _derivative(three, P, F, np.ascontiguousarray(attr[:, :3]), None, 301, 333, terms)
    _same(x, y[..., [0, 1, 2, 4]])
