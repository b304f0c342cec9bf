"""The per-view calls at the limits of their sizes: no view at all, fewer cameras or vertices than the renderer's buffers
hold, more than they hold."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2405_02508_gb300 import binding as B
from paper_2405_02508_gb300 import scenes
from paper_2405_02508_gb300.render import MerRender, Renderer

H, W = 60, 84


def _setup(views, n=8, **kw):
    P, F = scenes.octasphere(n)
    sh = scenes.Shading(n_main=3, C=4, mask_ch=3, bg=[0.1, 0.2, 0.3, 0.0])
    r = Renderer(torch.from_numpy(F.astype(np.int32)), len(P), views, H, W, sh, 3, **kw)
    verts = torch.from_numpy(P.astype(np.float32)).to(r.device)
    attr = torch.from_numpy(np.random.default_rng(n).uniform(0, 1, (len(P), 3)).astype(np.float32)).to(r.device)
    cams = B.cameras_tensor(scenes.cameras_on_sphere(max(views, 1), 3.0, H, W, 2), r.device)[:views]
    return r, verts, attr, cams


@pytest.mark.gpu
@pytest.mark.parametrize("zero", [0, 1, 2])
def test_no_views(zero):
    """Gradients over no view are zero where they are overwritten and left alone where they are added to."""
    r, verts, attr, cams = _setup(0)
    r.grad_verts.fill_(7.0)
    copy, ga = torch.full_like(r.grad_verts, 5.0), torch.full_like(attr, 7.0)
    r._backward(r.drawn(), torch.empty_like(r.image), cams, attr, None, r.terms, ga, copy, zero)
    assert (r.grad_verts == (0.0 if zero else 7.0)).all() and torch.equal(copy, r.grad_verts)
    assert (ga == (0.0 if zero == 2 else 7.0)).all()


@pytest.mark.gpu
def test_no_views_autograd():
    r, verts, attr, cams = _setup(0)
    v, a = verts.clone().requires_grad_(True), attr.clone().requires_grad_(True)
    image = MerRender.apply(v, a, None, cams, r)
    assert image.shape == (0, H, W, 4)
    stale = [torch.full_like(verts, float("nan")) for _ in range(8)]  # what the allocator hands out next
    del stale
    gv, ga = torch.autograd.grad(image, (v, a), torch.empty_like(image))
    assert (gv == 0).all() and (ga == 0).all()


@pytest.mark.gpu
@pytest.mark.parametrize("autograd", [False, True])
def test_fewer_cameras(autograd):
    """Two cameras on a renderer of three views: the two views and the gradient over them, as a renderer of two gives; the
    third view stays empty."""
    r, verts, attr, cams = _setup(3)
    two, _, _, _ = _setup(2)
    g = torch.randn(r.image.shape, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    r.terms = two.terms = 7 | B.MER_DETERMINISTIC
    ga, gt = torch.zeros_like(attr), torch.zeros_like(attr)
    two.forward(verts, cams[:2], attr)
    want = two.backward(g[:2].contiguous(), cams[:2], attr, terms=two.terms, grad_attr=gt)
    if autograd:
        v, a = verts.clone().requires_grad_(True), attr.clone().requires_grad_(True)
        image = MerRender.apply(v, a, None, cams[:2], r)
        got, ga = torch.autograd.grad(image, (v, a), g)
    else:
        image = r.forward(verts, cams[:2], attr)
        got = r.backward(g, cams[:2], attr, terms=r.terms, grad_attr=ga)
    assert torch.equal(image[:2], two.image) and (r.index[2] == -1).all()
    assert torch.equal(got, want) and torch.equal(ga, gt)
    t = torch.randn(verts.shape, generator=torch.Generator(device="cuda").manual_seed(2), device="cuda")
    d = r.forward_grad(t, cams[:2], attr)
    assert torch.equal(d[:2], two.forward_grad(t, cams[:2], attr)) and (d[2] == 0).all()


@pytest.mark.gpu
def test_fewer_vertices():
    """The first vertices moved on a renderer of two views: both views show them, the other vertices stay."""
    r, verts, attr, cams = _setup(2)
    few = len(verts) // 2
    moved = verts.clone()
    moved[:few] *= 1.1
    want = r.forward(moved, cams, attr).clone()
    r.forward(verts, cams, attr)
    assert torch.equal(r.forward(moved[:few], cams, attr), want)
    t = torch.zeros_like(verts)
    t[:few] = 1.0
    assert torch.equal(r.forward_grad(t[:few], cams, attr), r.forward_grad(t, cams, attr))
