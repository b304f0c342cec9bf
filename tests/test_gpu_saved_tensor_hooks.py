"""Hooks on the autograd function's saved tensors: what they give back in another type, place or layout is read as what it
holds, and gradients are those without hooks."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2405_02508_gb300 import binding as B
from paper_2405_02508_gb300 import scenes
from paper_2405_02508_gb300.render import MerRender, Renderer

pytestmark = pytest.mark.gpu

H, W, VIEWS = 60, 84, 2


def _spread(t):
    """The same values with a gap after each."""
    wide = torch.zeros((*t.shape, 2), dtype=t.dtype, device=t.device)
    wide[..., 0] = t
    return wide[..., 0]


PACKS = {
    "layout": (lambda t: t, lambda t: _spread(t)),
    "type": (lambda t: t, lambda t: t.double()),
    "place": (lambda t: t.cpu(), lambda t: t),
}


@pytest.mark.parametrize("how", sorted(PACKS))
def test_saved_drawing_through_hooks(how):
    P, F = scenes.octasphere(8)
    sh = scenes.Shading(n_main=3, C=4, mask_ch=3, bg=[0.1, 0.2, 0.3, 0.0])
    r = Renderer(torch.from_numpy(F.astype(np.int32)), len(P), VIEWS, H, W, sh, 3)
    r.terms = 7 | B.MER_DETERMINISTIC
    verts = torch.from_numpy(P.astype(np.float32)).cuda().requires_grad_(True)
    attr = torch.rand((len(P), 3), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda").requires_grad_(True)
    cams = B.cameras_tensor(scenes.cameras_on_sphere(VIEWS, 3.0, H, W, 2))
    g = torch.randn((VIEWS, H, W, 4), generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    want = torch.autograd.grad(MerRender.apply(verts, attr, None, cams, r), (verts, attr), g)
    pack, unpack = PACKS[how]
    drawn = {tuple(t.shape) for t in (r.vpix, r.index, r.image)}  # (the cover image has the shape of the index)

    def on(f):
        return lambda t: f(t) if tuple(t.shape) in drawn else t

    with torch.autograd.graph.saved_tensors_hooks(on(pack), on(unpack)):
        image = MerRender.apply(verts, attr, None, cams, r)
    got = torch.autograd.grad(image, (verts, attr), g)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
