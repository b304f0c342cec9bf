"""The whole-pass calls of the per-view path (mer_view_render, mer_view_backward, mer_view_forward_grad) against the stages
called one by one: the same images bit for bit, at sizes on both sides of the one-launch scan and of the clearing in the
projection; bin overflow, device errors, capture, and an autograd graph whose renderer draws something else in between."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2405_02508_gb300 import binding as B
from paper_2405_02508_gb300 import scenes
from paper_2405_02508_gb300.render import MerRender, Renderer

pytestmark = pytest.mark.gpu

SHADES = {
    "rgb": dict(n_main=3, C=3, bg=[0.5, 0.4, 0.3]),
    "normals": dict(n_main=3, C=5, mask_ch=3, depth_ch=4, bg=[0.1] * 5),
    "texture": dict(n_main=3, C=4, uv_offset=0, mask_ch=3, bg=[0.2] * 4),
    "generic": dict(n_main=2, C=4, mask_ch=3, backface_ch=2, bg=[0.2] * 4),
}


def _setup(shade, H, W, views, n=10, tile=16, precise=False):
    P, F = scenes.octasphere(n)
    rng = np.random.default_rng(n)
    sh = scenes.Shading(**SHADES[shade])
    attr = scenes.equirect_uv(P) if shade == "texture" else rng.uniform(0, 1, (len(P), 3))
    tex = torch.rand((16, 32, 4), generator=torch.Generator().manual_seed(1)).cuda() if shade == "texture" else None
    verts = torch.from_numpy(P.astype(np.float32)).cuda()
    cams = B.cameras_tensor(scenes.cameras_on_sphere(views, 3.0, H, W, 2))
    r = Renderer(torch.from_numpy(F.astype(np.int32)), len(P), views, H, W, sh, attr.shape[1],
                 None if tex is None else tex.shape, tile=tile, precise=precise)
    return r, verts, cams, torch.from_numpy(attr.astype(np.float32)).cuda(), tex


# 38,088 tiles: more than one CTA scans; 8 x 8 pixels: one tile; octasphere(1) at tile 8: many more tiles than vertices
@pytest.mark.parametrize("shade", sorted(SHADES))
@pytest.mark.parametrize("H,W,views,n,tile,precise", [(8, 8, 1, 3, 8, False), (61, 75, 3, 10, 16, False),
                                                      (1101, 1097, 2, 1, 8, False), (130, 70, 2, 8, 32, True)])
def test_passes_equal_stages(shade, H, W, views, n, tile, precise):
    r, verts, cams, attr, tex = _setup(shade, H, W, views, n, tile, precise)
    out = {}
    for whole in (False, True):
        depth = torch.full((views, H, W), -7.0, device="cuda")
        bary = torch.full((views, H, W, 2), -7.0, device="cuda")
        r.index.fill_(-9)
        r.image.fill_(-9.0)
        r.cover.fill_(255)
        r.vpix.zero_()
        copies = (torch.zeros_like(r.vpix), torch.zeros_like(r.index), torch.zeros_like(r.image))
        if whole:
            r.forward(verts, cams, attr, tex, depth, bary, copies=copies)
            for a, b in zip(copies, (r.vpix, r.index, r.image)):
                assert torch.equal(a.view(torch.int32), b.view(torch.int32))
        else:
            r.project(verts, cams)
            r.rasterize(depth, bary)
            r.shade(attr, tex)
        out[whole] = [t.clone() for t in (r.vpix.view(torch.int32), r.index, r.image, r.cover, depth, bary)]
        assert (r.index >= 0).any()
    for a, b in zip(out[False], out[True]):
        assert torch.equal(a, b)
    # gradients: the reproducible option, so that sums in another order do not matter
    g = torch.randn(r.image.shape, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    terms = 7 | B.MER_DETERMINISTIC
    ga = torch.zeros_like(attr)
    gv = r.backward(g, cams, attr, tex, terms=terms, grad_attr=ga).clone()
    gp = r.grad_vpix.clone()
    first = ga.clone()
    r.grad_vpix.zero_()
    r.grad_verts.zero_()
    gs = torch.zeros_like(attr)
    B.mer_backward(r.vpix, r.tris, r.index, r.image, g, attr, tex, r.sh, terms, r.grad_vpix, gs, r.workspace, r.cover)
    B.mer_project_backward(cams, r.vpix, r.grad_vpix, r.grad_verts)
    assert torch.equal(gp, r.grad_vpix) and torch.equal(gv, r.grad_verts) and torch.equal(first, gs)
    r.backward(g, cams, attr, tex, terms=terms, grad_attr=ga, zero=False)  # adds to what is there
    torch.testing.assert_close(r.grad_vpix, 2 * gp, rtol=1e-12, atol=0)
    t = torch.randn(verts.shape, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda")
    d = r.forward_grad(t, cams, attr, tex)
    tv = torch.empty((views, len(verts), 3), device="cuda")
    want = torch.empty_like(r.image)
    B.mer_project_jvp(t, cams, r.vpix, tv)
    B.mer_forward_grad(r.vpix, r.tris, r.index, r.image, tv, attr, tex, r.sh, 7, want, r.workspace)
    assert torch.equal(d, want)


def test_overflow_and_range_are_reported():
    r, verts, cams, attr, tex = _setup("normals", 200, 160, 1)
    want = r.forward(verts, cams, attr, tex).clone()
    small = B.mer_workspace_size(r.V, r.T, r.n, r.H, r.W, r.tile, 1)
    r.workspace = torch.zeros(small // 4 + 64, dtype=torch.float32, device="cuda")
    assert torch.equal(r.forward(verts, cams, attr, tex), want) and r.workspace.numel() > small // 4 + 64
    good = int(r.tris[5, 1])
    r.tris[5, 1] = r.V
    with pytest.raises(B.MerError) as e:
        r.forward(verts, cams, attr, tex)
    assert e.value.code == B.MER_ERANGE
    r.tris[5, 1] = good
    assert torch.equal(r.forward(verts, cams, attr, tex), want)  # the status word was cleared


def test_capture():
    r, verts, cams, attr, tex = _setup("texture", 90, 110, 2)
    want = r.forward(verts, cams, attr, tex).clone()
    g = torch.randn_like(r.image)
    r.backward(g, cams, attr, tex)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        r.forward(verts, cams, attr, tex, checked=False)
        r.backward(g, cams, attr, tex)
        with pytest.raises(B.MerError) as e:  # a capturing stream cannot be waited for
            r.forward(verts, cams, attr, tex)
        assert e.value.code == B.MER_ECUDA
    r.image.zero_()
    graph.replay()
    assert torch.equal(r.image, want)


def test_autograd_with_a_renderer_in_use():
    """Two graphs of one renderer, run backward in either order and after other work, give each its own gradients; both
    leave the returned images alone."""
    r, verts, cams, attr, tex = _setup("rgb", 120, 100, 2)
    r.terms = 7 | B.MER_DETERMINISTIC
    g = torch.randn_like(r.image)

    def graph(scale):
        v = (verts * scale).requires_grad_(True)
        a = attr.clone().requires_grad_(True)
        return MerRender.apply(v, a, tex, cams, r), v, a

    alone = []
    for scale in (1.0, 0.7):
        im, v, a = graph(scale)
        alone.append((im.detach().clone(), *torch.autograd.grad(im, (v, a), g)))
    for order in ((0, 1), (1, 0)):
        graphs = [graph(1.0), graph(0.7)]
        r.project(verts * 0.5, cams)
        r.rasterize()
        for k in order:
            im, v, a = graphs[k]
            got = torch.autograd.grad(im, (v, a), g)
            assert torch.equal(im, alone[k][0]) and torch.equal(got[0], alone[k][1]) and torch.equal(got[1], alone[k][2])
            assert torch.equal(r.image, im.detach())  # the renderer's buffers hold what was differentiated


def test_passes_back_to_back():
    """Passes queued without waiting, over two geometries in turn, each give what they give alone (a kernel of a pass is
    set up while the one before it runs, and must not read what that one has not written yet)."""
    r, verts, cams, attr, tex = _setup("texture", 301, 333, 2, n=40)
    g = torch.randn_like(r.image)
    sets = [verts, verts * 0.8]
    terms = 7 | B.MER_DETERMINISTIC

    def once(v):
        r.forward(v, cams, attr, tex, checked=False)
        gv = r.backward(g, cams, attr, tex, terms=terms)
        return r.image.clone(), r.index.clone(), gv.clone()

    alone = []
    for v in sets:
        torch.cuda.synchronize()
        alone.append(once(v))
        torch.cuda.synchronize()
    got = [once(sets[k % 2]) for k in range(40)]
    for k, out in enumerate(got):
        for a, b in zip(out, alone[k % 2]):
            assert torch.equal(a, b)


def test_forward_grad_keeps_nan():
    """A tangent that is not a number reaches every pixel whose pairs it moves."""
    r, verts, cams, attr, tex = _setup("rgb", 90, 110, 1)
    r.forward(verts, cams, attr, tex)
    t = torch.randn(verts.shape, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda")
    moved = r.forward_grad(t, cams, attr, tex, terms=B.MER_EDGE) != 0
    assert moved.any()
    assert torch.isnan(r.forward_grad(torch.full_like(t, float("nan")), cams, attr, tex, terms=B.MER_EDGE))[moved].all()
