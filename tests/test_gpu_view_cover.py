"""The cover image of the per-view path belongs to the drawing that is differentiated: with the ordinary (fast) backward,
which skips the pixel pairs that it rules out, gradients are those of a renderer without cover images, also when the renderer
has drawn something else in between, by a call or by a replayed graph."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2405_02508_gb300 import binding as B
from paper_2405_02508_gb300 import scenes
from paper_2405_02508_gb300.render import MerRender, Renderer

pytestmark = pytest.mark.gpu

H, W, VIEWS = 150, 187, 2


def _setup(tile=16):
    """Two spheres of which one is in front of the other (a), and side by side (b): a has pairs that scatter all over,
    and b's cover image rules most of them out."""
    P, F = scenes.octasphere(12)
    P = P.astype(np.float32)
    F = np.concatenate([F, F + len(P)]).astype(np.int32)
    near, apart = np.float32([[0.5, 0.3, 0.4]]), np.float32([[30.0, 0.0, 0.0]])
    a = torch.from_numpy(np.concatenate([P, 0.6 * P + near])).cuda()
    b = torch.from_numpy(np.concatenate([0.9 * P, 0.6 * P + apart])).cuda()
    attr = torch.from_numpy(np.random.default_rng(3).uniform(0, 1, (len(a), 3)).astype(np.float32)).cuda()
    cams = B.cameras_tensor(scenes.cameras_on_sphere(VIEWS, 4.0, H, W, 2))
    sh = scenes.Shading(n_main=3, C=4, mask_ch=3, bg=[0.1, 0.2, 0.3, 0.0])
    r, plain = (Renderer(torch.from_numpy(F), len(a), VIEWS, H, W, sh, 3, tile=tile, cover_hint=hint) for hint in (True, False))
    g = torch.randn((VIEWS, H, W, 4), generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    return r, plain, a, b, attr, cams, g


def _expected(plain, verts, attr, cams, g):
    ga = torch.zeros_like(attr)
    plain.forward(verts, cams, attr)
    gv = plain.backward(g, cams, attr, grad_attr=ga)
    return gv.clone(), ga


def _close(got, want):
    """The same FP32 terms summed in another order: within 2^-24 times the number of terms of a tile (at most 512) of the
    largest sum."""
    for x, y in zip(got, want):
        assert float((x - y).abs().max()) <= 512 * 2.0 ** -24 * float(y.abs().max())


def _apply(r, verts, attr, cams):
    v, a = verts.clone().requires_grad_(True), attr.clone().requires_grad_(True)
    return MerRender.apply(v, a, None, cams, r), v, a


@pytest.mark.parametrize("tile", [8, 16, 32])
def test_view_passes(tile):
    """One pass after another over the two geometries, queued without waiting, and through the autograd function."""
    r, plain, a, b, attr, cams, g = _setup(tile)
    want = [_expected(plain, v, attr, cams, g) for v in (a, b)]
    got = []
    for k in range(8):
        ga = torch.zeros_like(attr)
        r.forward((a, b)[k % 2], cams, attr, checked=False)
        got.append((r.backward(g, cams, attr, grad_attr=ga).clone(), ga))
    for k in range(8):
        _close(got[k], want[k % 2])
    for k, v in enumerate((a, b)):
        im, vv, aa = _apply(r, v, attr, cams)
        _close(torch.autograd.grad(im, (vv, aa), g), want[k])


@pytest.mark.parametrize("other", ["forward", "stages", "graph"])
def test_another_drawing_in_between(other):
    r, plain, a, b, attr, cams, g = _setup()
    want = _expected(plain, a, attr, cams, g)
    graph = torch.cuda.CUDAGraph()
    if other == "graph":
        r.forward(b, cams, attr)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            r.forward(b, cams, attr, checked=False)
    im, v, at = _apply(r, a, attr, cams)
    if other == "forward":
        r.forward(b, cams, attr)
    elif other == "stages":
        r.project(b, cams)
        r.rasterize()
        r.shade(attr, None)
    else:
        graph.replay()
    _close(torch.autograd.grad(im, (v, at), g), want)
    assert torch.equal(r.image, im.detach())  # the buffers hold what was differentiated, the cover image with them
    ga = torch.zeros_like(attr)
    _close((r.backward(g, cams, attr, grad_attr=ga), ga), want)


@pytest.mark.parametrize("precise", [False, True])
def test_cover_copy(precise):
    """The second copy of the cover image, on both routes that write it; refused without a cover image to copy."""
    r, plain, a, b, attr, cams, g = _setup()
    r.sh.precise = plain.sh.precise = int(precise)
    copies = [torch.zeros_like(t) for t in r.drawn()]
    r.cover.fill_(255)
    r.forward(a, cams, attr, copies=copies)
    for x, y in zip(copies, r.drawn()):
        assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))
    assert int(r.cover.max()) < 128 and int((r.cover & 7).max()) > 0
    with pytest.raises(B.MerError) as e:
        plain.forward(a, cams, attr, copies=copies)
    assert e.value.code == B.MER_EINVAL
