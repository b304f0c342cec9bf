"""Forward/backward calls over the C-ABI, and the ``torch.autograd.Function``.

``Renderer`` owns the caller-side buffers (workspace, vertex records, images)
for one mesh and a batch of views and makes the library calls, one per pass:

    forward : mer_view_render (mer_project -> mer_rasterize -> mer_shade)
    backward: mer_view_backward (mer_backward (edge + interior) -> mer_project_backward)

A small render is a few dozen microseconds on the device, less than the host took for a dozen calls
with their arguments; the stages stay available one by one (``project``, ``rasterize``, ``shade``).

With ``cover_hint`` (default) the rasterizer also writes the cover image (which facings cover each pixel
centre, one byte a pixel) and the backward uses it to skip pixel pairs that cannot scatter; the results are
the same without it.

``MerRender.apply(verts, attr, tex, cams, renderer, recompute_bary)`` exposes the
same as an autograd function whose backward is the micro-edge kernel (with the
renderer's ``terms``; with MER_DETERMINISTIC among them the gradients are bitwise
reproducible).  With
``recompute_bary`` the barycentric image is never stored (the backward always
re-derives barycentrics from the index image and the vertex records), which
saves 8 bytes per pixel of activation memory.
"""
from __future__ import annotations

import numpy as np
import torch

from . import binding as B


class Renderer:
    def __init__(self, tris: torch.Tensor, V: int, n_views: int, H: int, W: int, shading, C_attr: int,
                 tex_shape=None, tile: int = 16, device: str = "cuda", cover_hint: bool = True,
                 precise: bool = False):
        """precise: FP64 shading rounded once per value (the image a MER_DETERMINISTIC backward expects).
        ``terms`` (attribute): the backward terms MerRender uses."""
        self.tris = tris.to(device=device, dtype=torch.int32).contiguous()
        self.T = int(self.tris.shape[0])
        self.V, self.n, self.H, self.W = int(V), int(n_views), int(H), int(W)
        self.tile = tile
        self.device = device
        self.shading = shading
        self.C = shading.C
        self.sh = B.shading_struct(shading, C_attr, None, precise)
        if tex_shape is not None:
            self.sh.tex_h, self.sh.tex_w = int(tex_shape[0]), int(tex_shape[1])
            self.sh.tex_c = int(tex_shape[2]) if len(tex_shape) > 2 else shading.n_main
        self.bg = shading.bg_array()
        n, H, W = self.n, self.H, self.W
        self.vpix = torch.zeros((n, self.V, B.VERTEX_FLOATS), dtype=torch.float32, device=device)  # (nothing in front)
        self.index = torch.empty((n, H, W), dtype=torch.int32, device=device)
        self.image = torch.empty((n, H, W, self.C), dtype=torch.float32, device=device)
        self.cover = torch.empty((n, H, W), dtype=torch.uint8, device=device) if cover_hint else None
        self.grad_vpix = torch.zeros((n, self.V, 3), dtype=torch.float64, device=device)
        self.grad_verts = torch.zeros((self.V, 3), dtype=torch.float32, device=device)
        self.terms = B.MER_EDGE | B.MER_INTERIOR | B.MER_INTERSECT
        self.renders = 0      # times the buffers were drawn to
        self.replayed = False  # drawn to under capture: replays draw again without being counted
        self._status = None   # pinned words the device reports the binning's status in (made by the first checked pass)
        self._alloc_workspace(0)

    def _alloc_workspace(self, capacity: int, at_least: int = 0):
        nbytes = max(B.mer_workspace_size(self.V, self.T, self.n, self.H, self.W, self.tile, capacity), at_least)
        self.workspace = torch.zeros((nbytes + 255) // 256 * 64, dtype=torch.float32, device=self.device)

    def _ensure_backward_workspace(self, terms: int, grad_attr):
        need = B.mer_backward_workspace_size(self.n * self.V, self.V, B.attr_grad_channels(self.sh, grad_attr), terms)
        if self.workspace.numel() * 4 < need:  # the raster's bins are not needed any more at this point
            self._alloc_workspace(0, need)

    # -- forward -----------------------------------------------------------------------------------
    def project(self, verts: torch.Tensor, cams: torch.Tensor):
        """Fewer vertices or cameras than the buffers hold give the first records of the first views; the others stay."""
        self._check_sizes(verts.shape[0], cams.shape[0])
        self._drawing()
        verts = verts.contiguous()
        if verts.shape[0] == self.V:
            B.mer_project(verts, cams, self.vpix)
            return
        for k in range(cams.shape[0]):  # a view's records start at a multiple of V
            B.mer_project(verts, cams[k:k + 1], self.vpix[k:k + 1])

    def project_screen(self, scr: torch.Tensor):
        """As ``project``, from screen positions [views, vertices, 3]."""
        self._check_sizes(scr.shape[1], scr.shape[0])
        self._drawing()
        scr = scr.contiguous()
        if scr.shape[1] == self.V:
            B.mer_project_screen(scr, self.vpix)
            return
        for k in range(scr.shape[0]):
            B.mer_project_screen(scr[k:k + 1], self.vpix[k:k + 1])

    def _check_sizes(self, V: int, n: int):
        if V > self.V or n > self.n:
            raise ValueError(f"{n} views of {V} vertices for a renderer of {self.n} views of {self.V}")

    def rasterize(self, depth: torch.Tensor | None = None, bary: torch.Tensor | None = None, checked: bool = True):
        self._drawing()
        B.mer_rasterize(self.vpix, self.tris, self.H, self.W, self.tile, self.workspace, self.index, depth, bary,
                        self.cover)
        if checked:
            code, total = B.mer_sync_status(self.workspace)
            if code == B.MER_EOVERFLOW:  # size the bin list exactly and redo
                self._alloc_workspace(int(total * 1.25) + 1024)
                B.mer_rasterize(self.vpix, self.tris, self.H, self.W, self.tile, self.workspace, self.index, depth,
                                bary, self.cover)
                code, total = B.mer_sync_status(self.workspace)
            if code != B.MER_OK:
                raise B.MerError(code, "mer_rasterize")

    def shade(self, attr: torch.Tensor, tex: torch.Tensor | None):
        self._drawing()
        B.mer_shade(self.vpix, self.tris, self.index, attr.contiguous(), tex, self.bg, self.sh, self.image,
                    self.workspace)

    def drawn(self) -> tuple:
        """The buffers that a backward pass reads: vertex records, index, image and cover image (or None)."""
        return self.vpix, self.index, self.image, self.cover

    def _drawing(self):
        self.renders += 1
        if not self.replayed and torch.cuda.is_current_stream_capturing():
            self.replayed = True

    def _view(self, bg=None) -> B.MerView:
        """The renderer's buffers for one call."""
        return B.view_struct(self.tris, self.V, self.n, self.H, self.W, self.tile, self.workspace, self.vpix, self.index,
                             self.cover, self.image, self.sh, bg)

    def forward(self, verts, cams, attr, tex=None, depth=None, bary=None, checked=True, copies=None):
        """copies (optional): (vpix, index, image) or (vpix, index, image, cover) tensors that receive second copies of
        those buffers."""
        if verts.shape[0] != self.V or cams.shape[0] != self.n:  # fewer vertices or cameras than the buffers hold
            self.project(verts, cams)
            self.rasterize(depth, bary, checked)
            self.shade(attr, tex)
            if copies is not None:
                for dst, src in zip(copies, (self.vpix, self.index, self.image, self.cover)):
                    dst.copy_(src)
            return self.image
        status = None
        if checked:
            if self._status is None:
                self._status = torch.zeros(2, dtype=torch.int64, pin_memory=True)
            status = self._status
            self.renders += 1
        else:
            self._drawing()
        verts, attr = verts.contiguous(), attr.contiguous()
        args = (verts, cams, attr, tex, depth, bary, copies or (None, None, None), status)
        code, total = B.mer_view_render(self._view(self.bg), *args)
        if code == B.MER_EOVERFLOW:  # size the bin list exactly and redo
            self._alloc_workspace(int(total * 1.25) + 1024)
            code, total = B.mer_view_render(self._view(self.bg), *args)
        if code != B.MER_OK:
            raise B.MerError(code, "mer_rasterize")
        return self.image

    # -- backward ----------------------------------------------------------------------------------
    def backward(self, grad_image: torch.Tensor, cams: torch.Tensor, attr: torch.Tensor, tex=None,
                 terms: int = B.MER_EDGE | B.MER_INTERIOR | B.MER_INTERSECT, grad_attr=None, zero: bool = True):
        return self._backward(self.drawn(), grad_image, cams, attr, tex, terms, grad_attr, None, int(bool(zero)))

    def _backward(self, drawn, grad_image, cams, attr, tex, terms, grad_attr, grad_verts_copy, zero):
        """drawn: the vpix, index, image and cover (if any) that the gradient is of; zero: 0, 1 or 2 as in
        mer_view_backward.  With fewer cameras than views, the vertex gradient is of the views that have one."""
        vpix, index, image, *cover = drawn
        cover = cover[0] if cover else None
        grad_image, attr = grad_image.contiguous(), attr.contiguous()
        if terms & B.MER_DETERMINISTIC:
            self._ensure_backward_workspace(terms, grad_attr)
        if cams.shape[0] >= self.n:
            view = B.view_struct(self.tris, self.V, self.n, self.H, self.W, self.tile, self.workspace, vpix, index, cover,
                                 image, self.sh)
            B.mer_view_backward(view, cams, grad_image, attr, tex, terms, self.grad_vpix, grad_attr, self.grad_verts,
                                grad_verts_copy, zero)
            return self.grad_verts
        if zero:
            self.grad_vpix.zero_()
            self.grad_verts.zero_()
        if zero > 1 and grad_attr is not None:
            grad_attr.zero_()
        B.mer_backward(vpix, self.tris, index, image, grad_image, attr, tex, self.sh, terms, self.grad_vpix, grad_attr,
                       self.workspace, cover)
        B.mer_project_backward(cams, vpix, self.grad_vpix, self.grad_verts)
        if grad_verts_copy is not None:
            grad_verts_copy.copy_(self.grad_verts)
        return self.grad_verts

    # -- forward gradients ---------------------------------------------------------------------------
    def forward_grad(self, tangent_world: torch.Tensor, cams: torch.Tensor, attr: torch.Tensor, tex=None,
                     terms: int = B.MER_EDGE | B.MER_INTERIOR | B.MER_INTERSECT) -> torch.Tensor:
        """d(image)/d(theta) [n,H,W,C] for a world-space vertex tangent [V,3] (after ``forward``).  Vertices without a
        tangent and views without a camera (fewer than the buffers hold) do not move."""
        out = torch.empty_like(self.image)
        if tangent_world.shape[0] < self.V or cams.shape[0] < self.n:
            tv = torch.zeros((self.n, self.V, 3), dtype=torch.float32, device=self.device)
            moved = torch.zeros((self.V, 3), dtype=torch.float32, device=self.device)
            moved[:tangent_world.shape[0]] = tangent_world[:self.V]
            B.mer_project_jvp(moved, cams, self.vpix, tv)
            B.mer_forward_grad(self.vpix, self.tris, self.index, self.image, tv, attr.contiguous(), tex, self.sh, terms,
                               out, self.workspace)
            return out
        tv = torch.empty((self.n, self.V, 3), dtype=torch.float32, device=self.device)
        B.mer_view_forward_grad(self._view(), cams, tangent_world.contiguous(), attr.contiguous(), tex, terms, tv, out)
        return out

    def check_status(self):
        code, _ = B.mer_sync_status(self.workspace)
        if code != B.MER_OK:
            raise B.MerError(code, "device status")


def _as_buffer(t: torch.Tensor, like: torch.Tensor | None) -> torch.Tensor:
    """A saved tensor as the kernels read it: a hook on saved tensors may give it back in another type, place or layout."""
    if like is None or (t.dtype == like.dtype and t.shape == like.shape and t.device == like.device and t.is_contiguous()):
        return t
    return torch.empty_like(like).copy_(t)


class MerRender(torch.autograd.Function):
    """image = render(verts, attr); backward = micro-edge + interior kernels.

    ``verts`` [V,3] and ``attr`` [V,C_attr] are differentiable; ``tex`` and the
    cameras are not.  The renderer's shading program decides the channels.
    """

    @staticmethod
    def forward(ctx, verts, attr, tex, cams, renderer: Renderer, recompute_bary: bool = True):
        r = renderer
        bary = None
        if not recompute_bary:
            bary = torch.empty((r.n, r.H, r.W, 2), dtype=torch.float32, device=r.device)
        # the gradient is of this drawing, whatever the renderer's buffers hold by then (another forward, a replayed graph)
        saved = [torch.empty_like(t) for t in r.drawn() if t is not None]
        r.forward(verts, cams, attr, tex, bary=bary, copies=saved)
        ctx.renderer = r
        ctx.renders = r.renders
        ctx.save_for_backward(verts, attr, cams, tex, bary, *saved)
        return saved[2]

    @staticmethod
    def backward(ctx, grad_image):
        r = ctx.renderer
        verts, attr, cams, tex, _, *saved = ctx.saved_tensors
        saved = [_as_buffer(t, like) for t, like in zip(saved, r.drawn())]
        if r.renders != ctx.renders or r.replayed:  # the buffers hold another drawing: put back what is differentiated
            for dst, src in zip(r.drawn(), saved):
                if dst is not None:
                    dst.copy_(src)
            r.renders += 1
        grad_attr, zero = None, 1
        if ctx.needs_input_grad[1]:
            if attr.shape == (r.V, r.sh.C_attr):
                grad_attr, zero = torch.empty_like(attr), 2
            else:
                grad_attr = torch.zeros_like(attr)
        gv = torch.empty_like(r.grad_verts)
        r._backward(saved, grad_image, cams, attr, tex, r.terms, grad_attr, gv, zero)
        return gv, grad_attr, None, None, None, None
