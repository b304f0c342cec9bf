"""The per-view calls with fewer cameras or vertices than the renderer's buffers hold: what reaches the library stays inside
the tensors, and a view's records start where the raster reads them; more than the buffers hold is refused.  Host logic, with a
stand-in for the library that works on host memory."""
from __future__ import annotations

import ctypes

import pytest
import torch

from paper_2405_02508_gb300 import binding as B
from paper_2405_02508_gb300 import scenes
from paper_2405_02508_gb300.render import Renderer

V, N, H, W = 7, 3, 16, 24


class _Library:
    """mer_project marks each record it writes; the calls that read cameras note how many they read, and the rows."""

    def __init__(self):
        self.calls = []

    def mer_project(self, verts, V_, cams, n, vpix, stream):
        if n * V_ > N * V:  # (the real one would write past the records)
            return B.MER_EINVAL
        for i in range(n * V_):
            ctypes.c_int32.from_address(vpix + i * 4 * B.VERTEX_FLOATS).value = 1000 + i % V_
        self.calls.append(("mer_project", n, V_))
        return 0

    def mer_project_screen(self, scr, V_, n, vpix, stream):
        return self.mer_project(scr, V_, None, n, vpix, stream)

    def __getattr__(self, name):
        if name == "mer_workspace_size":
            return lambda *a: 4096
        if name == "mer_backward_workspace_size":
            return lambda *a: 256

        def call(*a):
            if name == "mer_project_backward":
                self.calls.append((name, a[2], a[0]))
            elif name == "mer_project_jvp":
                self.calls.append((name, a[3], a[1]))
            elif name == "mer_rasterize_world":
                self.calls.append((name, a[5], a[1]))
            elif name in ("mer_view_backward", "mer_view_forward_grad", "mer_view_render", "mer_view_render_cover"):
                v = a[0]
                self.calls.append((name, v.n, v.V))
            return 0

        return call

    def cameras_read(self):
        return max([n for name, n, _ in self.calls], default=0)


@pytest.fixture
def lib(monkeypatch):
    fake = _Library()
    monkeypatch.setattr(B, "lib", lambda *a: fake)
    monkeypatch.setattr(B, "_ptr", lambda t: None if t is None else t.data_ptr())
    monkeypatch.setattr(B, "_stream", lambda: None)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    return fake


def _renderer():
    sh = scenes.Shading(n_main=3, C=3, bg=[0.0] * 3)
    return Renderer(torch.zeros((4, 3), dtype=torch.int32), V, N, H, W, sh, 3, device="cpu")


def _cams(n):
    return torch.zeros((n, B.CAMERA_DOUBLES), dtype=torch.float64)


@pytest.mark.parametrize("screen", [False, True])
@pytest.mark.parametrize("v,n", [(V, N), (V, 2), (V, 0), (5, N), (5, 2), (5, 1), (0, 2)])
def test_records_at_the_views_stride(lib, v, n, screen):
    r = _renderer()
    r.vpix.zero_()
    if screen:
        r.project_screen(torch.zeros((n, v, 3), dtype=torch.float64))
    else:
        r.project(torch.zeros((v, 3)), _cams(n))
    want = torch.zeros((N, V), dtype=torch.int32)
    want[:n, :v] = 1000 + torch.arange(v, dtype=torch.int32)
    assert torch.equal(r.vpix.view(torch.int32)[..., 0], want)


@pytest.mark.parametrize("v,n", [(V + 1, 1), (V, N + 1), (V + 1, N)])
def test_more_than_the_buffers_hold(lib, v, n):
    r = _renderer()
    with pytest.raises(ValueError, match="vertices"):
        r.project(torch.zeros((v, 3)), _cams(n))
    with pytest.raises(ValueError, match="vertices"):
        r.forward(torch.zeros((v, 3)), _cams(n), torch.zeros((V, 3)), checked=False)
    with pytest.raises(ValueError, match="vertices"):
        r.project_screen(torch.zeros((n, v, 3), dtype=torch.float64))
    with pytest.raises(ValueError, match="do not fit"):
        B.mer_project(torch.zeros((v, 3)), _cams(n), torch.zeros((n, v, B.VERTEX_FLOATS - 1)))
    assert not lib.calls


@pytest.mark.parametrize("n", [1, 2])
def test_no_more_cameras_read_than_given(lib, n):
    r = _renderer()
    attr, cams = torch.zeros((V, 3)), _cams(n)
    g = torch.zeros((N, H, W, 3))
    r.backward(g, cams, attr)
    r._backward(r.drawn(), g, cams, attr, None, r.terms, torch.zeros_like(attr), torch.zeros((V, 3)), 2)
    r.forward_grad(torch.zeros((V, 3)), cams, attr)
    B.mer_project_backward(cams, r.vpix, r.grad_vpix, r.grad_verts)
    B.mer_project_jvp(torch.zeros((V, 3)), cams, r.vpix, torch.zeros((N, V, 3)))
    assert 0 < lib.cameras_read() <= n
    with pytest.raises(ValueError, match="records"):
        B.mer_rasterize_world(torch.zeros((V, 3)), r.tris, cams, H, W, 16, r.workspace, r.index, r.vpix)


def test_no_more_tangents_read_than_given(lib, monkeypatch):
    r = _renderer()
    seen, real = [], B.mer_project_jvp
    monkeypatch.setattr(B, "mer_project_jvp", lambda t, *a: (seen.append(t.shape[0]), real(t, *a)))
    r.forward_grad(torch.ones((V - 2, 3)), _cams(N), torch.zeros((V, 3)))
    assert seen == [V]
    with pytest.raises(ValueError, match="tangent"):
        real(torch.zeros((V - 1, 3)), _cams(N), r.vpix, torch.zeros((N, V, 3)))
