"""Performance cases of the micro-edge rasterizer: what a user's program has it do, over the sizes it is used at.

Every case goes through a public entry point of the package: the autograd function (``MerRender``), the per-view
renderer (``Renderer``), the batched renderer as a captured step (``BatchRenderer``), the uneven fitting loop's
gradient (``UnevenFit``), the Laplacian preconditioner, forward gradients and the deterministic option.  Meshes,
cameras, textures and upstream gradients are drawn from the seed, with the shapes of the repository's own scenes.

``exact`` computes the same results in 64 bits with plain torch: coverage with integers, depth, shading and the
interior gradient by torch's autograd, the micro-edge term (Eq. 11, the Sec. 4.3 rule, Eq. 12) spelled out.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2405_02508_gb300 import binding as B
from paper_2405_02508_gb300 import scenes
from paper_2405_02508_gb300.batch import BatchRenderer
from paper_2405_02508_gb300.fit import UnevenFit
from paper_2405_02508_gb300.precond import LaplacianPreconditioner
from paper_2405_02508_gb300.render import MerRender, Renderer

DEV = "cuda"
FIT_SIGMA = 0.002  # position noise of the fitting case
ALL_TERMS = B.MER_EDGE | B.MER_INTERIOR | B.MER_INTERSECT

# Image layouts: interpolated colours, normals with mask and depth, textured with mask (and depth), normals with mask.
SHADINGS = {
    "rgb": dict(n_main=3, C=3, bg=[0.5, 0.5, 0.5]),
    "normals": dict(n_main=3, C=5, mask_ch=3, depth_ch=4, bg=[0.0] * 5),
    "texture": dict(n_main=3, C=4, uv_offset=0, mask_ch=3, bg=[0.0] * 4),
    "texture_depth": dict(n_main=3, C=5, uv_offset=0, mask_ch=3, depth_ch=4, bg=[0.0] * 5),
    "normals_mask": dict(n_main=3, C=4, mask_ch=3, bg=[0.0] * 4),
}


def listed():
    return [
        # The smallest call: a 1,280-triangle mesh at 128 x 128 through the autograd function, as a toy fit does per step.
        dict(name="autograd_icosphere_128", kind="autograd", mesh="icosphere", n=3, views=1, H=128, W=128, shade="rgb"),
        # One view of two intersecting meshes with normals, mask and depth: an ordinary geometry-supervised step.
        dict(name="view_two_spheres_512", kind="view", mesh="pair", n=5, views=1, H=512, W=512, shade="normals"),
        # One textured head-scale view with gradients to the positions and the texture coordinates.
        dict(name="autograd_head_1024", kind="autograd", mesh="octasphere", n=128, views=1, H=1024, W=1024,
             shade="texture"),
        # A few views of a mid-size mesh at an odd image size.
        dict(name="view_ragged_333x517", kind="view", mesh="octasphere", n=40, views=3, H=333, W=517, shade="normals"),
        # A handful of moderate views per step through the batched path, recorded as a graph.
        dict(name="graph_8x512", kind="graph", mesh="octasphere", n=64, views=8, H=512, W=512, shade="texture_depth",
             tile=32),
        # Multi-view head reconstruction: 32 full-size views of the 131,072-triangle mesh per step, the largest case.
        dict(name="graph_head_32x1334x2048", kind="graph", mesh="octasphere", n=128, views=32, H=2048, W=1334,
             shade="texture_depth", tile=64),
        # The gradient of the uneven-batch fit: many meshes of 500 to 200k triangles at 128 to 1024 square, one view each,
        # positions near their targets (noise well below the edge length: the finest meshes do not fold over).
        dict(name="fit_uneven_48", kind="fit", items=48),
        # The preconditioner's solve (two per step of the preconditioned fit) on the head mesh, and on a small mesh.
        dict(name="solve_head", kind="solve", mesh="octasphere", n=128, lam=16.0),
        dict(name="solve_icosphere", kind="solve", mesh="icosphere", n=3, lam=16.0),
        # The derivative image along a vertex motion, for inspecting a parameter.
        dict(name="forward_grad_512", kind="jvp", mesh="octasphere", n=64, views=1, H=512, W=512, shade="texture"),
        # Reproducible training: FP64 shading and bitwise reproducible gradients.
        dict(name="deterministic_512", kind="det", mesh="pair", n=5, views=1, H=512, W=512, shade="normals"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["autograd", "view", "graph", "graph", "fit", "solve", "jvp", "det"])
    if kind == "fit":
        return dict(kind=kind, items=_log(rng, 2, 48))
    if kind == "solve":
        return dict(kind=kind, mesh="octasphere", n=_log(rng, 8, 128), lam=float(rng.choice([8, 16, 32])))
    top = {"autograd": 1024, "view": 1024, "graph": 2048, "jvp": 768, "det": 640}[kind]
    H, W = _log(rng, 64, top), _log(rng, 64, top)
    views = 1
    if kind == "view":
        views = rng.randint(1, 4)
    elif kind == "graph":
        views = min(_log(rng, 1, 32), max(1, 87_000_000 // (H * W)))
    shade = rng.choice(["rgb", "normals", "texture"] if kind == "autograd" else
                       ["rgb", "normals", "texture", "texture_depth", "normals_mask"])
    if kind in ("view", "det") and rng.random() < 0.3:
        mesh, n = "pair", rng.randint(3, 5)
    else:  # down to about one triangle a pixel
        mesh, n = "octasphere", _log(rng, 8, max(12, min(128, int(math.sqrt(H * W / 8)))))
    case = dict(kind=kind, mesh=mesh, n=n, views=views, H=H, W=W, shade=shade)
    if kind == "graph":
        case["tile"] = rng.choice([16, 32, 64])
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=128)
def _unit(mesh, n):
    """The undisplaced mesh: unit directions and triangles (topology does not depend on the seed)."""
    P, F = scenes.icosphere(n) if mesh in ("icosphere", "pair") else scenes.octasphere(n)
    return torch.from_numpy(P), torch.from_numpy(F.astype(np.int32))


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _mesh(mesh, n, seed):
    """Positions [V,3] float32 and triangles: a sphere displaced by a random smooth field and a little noise, or two
    jittered intersecting spheres."""
    P, F = _unit(mesh, n)
    P, F = P.to(DEV), F.to(DEV)
    g = _gen(seed)
    if mesh == "pair":
        off = 0.3 / math.sqrt(3.0)
        v = torch.cat([P + off, P - off])
        F = torch.cat([F, F + len(P)])
        v = v + 0.002 * torch.randn(v.shape, generator=g, device=DEV, dtype=torch.float64)
        return v.float(), F.contiguous()
    pw = [torch.ones_like(P)]
    for _ in range(4):
        pw.append(pw[-1] * P)
    mono = torch.stack([pw[a][:, 0] * pw[b][:, 1] * pw[c][:, 2]
                        for a in range(5) for b in range(5 - a) for c in range(5 - a - b)])
    s = torch.randn(len(mono), generator=g, device=DEV, dtype=torch.float64) @ mono
    s = s - s.mean()
    s = s / s.abs().max()
    r = 1.0 + 0.1 * s + 0.005 * torch.randn(len(P), generator=g, device=DEV, dtype=torch.float64)
    return (P * r[:, None]).float(), F.contiguous()


def _normals(v, tris):
    """Area-weighted unit normals, differentiable."""
    t = tris.long()
    a, b, c = v[t[:, 0]], v[t[:, 1]], v[t[:, 2]]
    fn = torch.linalg.cross(b - a, c - a)
    vn = torch.zeros_like(v)
    for k in range(3):
        vn = vn.index_add(0, t[:, k], fn)
    return vn / vn.norm(dim=1, keepdim=True)


def _texture(size, seed):
    """Smooth random RGB texture in [0, 1], padded to four floats a texel."""
    t = torch.rand((3, size, size), generator=_gen(seed), device=DEV)
    k = torch.fft.fftfreq(size, device=DEV)
    blur = torch.exp(-2.0 * (math.pi * 4.0) ** 2 * (k[:, None] ** 2 + k[None, :] ** 2))
    t = torch.fft.ifft2(torch.fft.fft2(t) * blur).real
    lo, hi = t.amin(dim=(1, 2), keepdim=True), t.amax(dim=(1, 2), keepdim=True)
    out = torch.zeros((size, size, 4), device=DEV)
    out[..., :3] = ((t - lo) / (hi - lo)).permute(1, 2, 0)
    return out


def _scene(case, seed):
    """Everything a renderer case needs but the upstream gradient."""
    verts, tris = _mesh(case["mesh"], case["n"], seed)
    sh = scenes.Shading(**SHADINGS[case["shade"]])
    tex = None
    if sh.uv_offset >= 0:
        P = _unit(case["mesh"], case["n"])[0].numpy()
        uv = scenes.equirect_uv(np.concatenate([P, P]) if case["mesh"] == "pair" else P)
        attr = torch.from_numpy(uv.astype(np.float32)).to(DEV)
        tex = _texture(1024 if case["n"] >= 64 else 256, seed + 1)
    elif case["shade"] == "rgb":
        attr = torch.rand(verts.shape, generator=_gen(seed + 2), device=DEV)
    else:
        attr = _normals(verts.double(), tris).float()
    radius = 4.5 if case["mesh"] == "pair" else 3.0
    cams = scenes.cameras_on_sphere(case["views"], radius, case["H"], case["W"], seed)
    return verts, tris, sh, attr, tex, cams


def _upstream(case, C, seed):
    return torch.randn((case["views"], case["H"], case["W"], C), generator=_gen(seed + 3), device=DEV)


def _tangent(verts, seed):
    return torch.randn(verts.shape, generator=_gen(seed + 4), device=DEV)


def _fit_items(case, seed):
    """Sizes as the uneven batch draws them (log-uniform triangles, four resolutions), the same for every seed, so
    that a case always costs the same; shapes and cameras from the seed."""
    ns, res = scenes.uneven_plan(case["items"])
    items = []
    for k, (n, r) in enumerate(zip(ns, res)):
        n = 8 * max(1, round(n / 8))  # a few frequencies, so that topology is built once
        v, t = _mesh("octasphere", n, 1000 * seed + k)
        cam = scenes.random_direction_camera(3.0, r, r, np.random.default_rng([seed, k]))
        items.append(scenes.Scene(f"item{k}", v.cpu().numpy(), t.cpu().numpy(), np.stack([cam]), r, r,
                                  np.zeros((len(v), 3), np.float32), scenes.Shading(**SHADINGS["normals_mask"])))
    return items


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fit":
        fit = UnevenFit(_fit_items(case, seed), sigma=FIT_SIGMA, seed=seed)
        return dict(kind=kind, fit=fit, x=fit.v_init)
    if kind == "solve":
        v, t = _mesh(case["mesh"], case["n"], seed)
        P = LaplacianPreconditioner(t.cpu().numpy(), len(v), case["lam"])
        return dict(kind=kind, P=P, b=torch.randn(v.shape, generator=_gen(seed + 5), device=DEV))
    verts, tris, sh, attr, tex, cams = _scene(case, seed)
    H, W, n = case["H"], case["W"], case["views"]
    s = dict(kind=kind, verts=verts, attr=attr, tex=tex)
    if kind != "jvp":
        s["grad"] = _upstream(case, sh.C, seed)
    if kind == "graph":
        mesh = (verts.cpu().numpy(), tris.cpu().numpy())
        br = BatchRenderer([mesh], [(0, k, H, W) for k in range(n)], cams, sh, attr.shape[1], tex, tile=case["tile"])
        br.prepare(verts, attr, tex)
        s["grad"] = s["grad"].view(-1, sh.C)
        br.capture(verts, attr, s["grad"], tex)
        s["br"] = br
        return s
    s["cams"] = B.cameras_tensor(cams)
    s["r"] = Renderer(tris, len(verts), n, H, W, sh, attr.shape[1], None if tex is None else tex.shape,
                      precise=kind == "det")
    if kind == "autograd":
        s["verts"] = verts.clone().requires_grad_(True)
        s["attr"] = attr.clone().requires_grad_(True)
    if kind == "jvp":  # the image is in hand; the derivative along the motion is what is asked for
        s["r"].forward(verts, s["cams"], attr, tex)
        s["tangent"] = _tangent(verts, seed)
    return s


def run(state):
    kind = state["kind"]
    if kind == "fit":
        g = state["fit"].loss_grad(state["x"])
        br = state["fit"].br
        return dict(image=br.image, index=br.index, grad_verts=g)
    if kind == "solve":
        return dict(x=state["P"].solve(state["b"]))
    if kind == "graph":
        br = state["br"]
        br.replay()
        return dict(image=br.image, index=br.index, grad_verts=br.grad_verts)
    r, cams, tex = state["r"], state["cams"], state["tex"]
    verts, attr = state["verts"], state["attr"]
    if kind == "autograd":
        image = MerRender.apply(verts, attr, tex, cams, r)
        gv, ga = torch.autograd.grad(image, (verts, attr), state["grad"])
        return dict(image=image, grad_verts=gv, grad_attr=ga)
    if kind == "jvp":
        return dict(derivative=r.forward_grad(state["tangent"], cams, attr, tex))
    r.forward(verts, cams, attr, tex)
    terms = ALL_TERMS | (B.MER_DETERMINISTIC if kind == "det" else 0)
    g = r.backward(state["grad"], cams, attr, tex, terms=terms)
    return dict(image=r.image, index=r.index, grad_verts=g)


def work(case):
    """Bytes: the mesh, attributes, texture and upstream gradient read once, image, index and gradients written once.
    Flops: about 100 a pixel to shade (barycentrics, interpolation), 150 to differentiate."""
    kind = case["kind"]
    if kind == "fit":
        ns, res = scenes.uneven_plan(case["items"])
        ns = [8 * max(1, round(n / 8)) for n in ns]
        px, V, T = sum(r * r for r in res), sum(4 * n * n + 2 for n in ns), sum(8 * n * n for n in ns)
        return dict(bytes=px * (4 + 2 * 16) + T * 12 + V * 24, flops=px * 250 + T * 60)
    n = case["n"]
    V, T = (4 * n * n + 2, 8 * n * n) if case["mesh"] == "octasphere" else (10 * 4 ** n + 2, 20 * 4 ** n)
    if case["mesh"] == "pair":
        V, T = 2 * V, 2 * T
    if kind == "solve":
        # edge graph, right-hand side and solution; conjugate gradients' own bound on the iterations for a 1e-6 residual
        its = 0.5 * math.sqrt(1.0 + 12.0 * case["lam"]) * math.log(2e6)
        return dict(bytes=8 * V + 4 * 2 * 1.5 * T + 24 * V, flops=its * V * 3 * 22)
    sh = SHADINGS[case["shade"]]
    tex = 16 * (1024 if n >= 64 else 256) ** 2 if "uv_offset" in sh else 0
    px, C, Ca = case["views"] * case["H"] * case["W"], sh["C"], 2 if "uv_offset" in sh else 3
    mesh = 12 * T + V * (12 + 4 * Ca) + tex + 136 * case["views"]
    if kind == "jvp":
        return dict(bytes=px * (4 + 8 * C) + mesh + 12 * V, flops=px * 150)
    ga = 4 * Ca * V if kind == "autograd" else 0
    return dict(bytes=px * (8 * C + (0 if kind == "autograd" else 4)) + mesh + 12 * V + ga, flops=px * 250)


# ---------------------------------------------------------------------------
# the same in 64 bits, with plain torch
# ---------------------------------------------------------------------------

def _project64(verts, cam):
    """Screen x, y and 1/Z of every vertex [V,3]; each operation rounded by itself, in the order the library states."""
    x, y, z = verts.double().unbind(1)
    R, t = [float(v) for v in cam["R"]], [float(v) for v in cam["t"]]
    X, Y, Z = (((R[3 * i] * x) + (R[3 * i + 1] * y)) + (R[3 * i + 2] * z) + t[i] for i in range(3))
    zeta = 1.0 / Z
    return torch.stack([float(cam["fx"]) * X * zeta + float(cam["cx"]), float(cam["fy"]) * Y * zeta + float(cam["cy"]),
                        zeta], 1)


def _edges(S, px, py):
    """The three integer edge functions of snapped triangles S [m,3,2] at snapped points (px, py)."""
    dx, dy = S[..., 0] - px[:, None], S[..., 1] - py[:, None]
    return torch.stack([dx[:, (i + 1) % 3] * dy[:, (i + 2) % 3] - dy[:, (i + 1) % 3] * dx[:, (i + 2) % 3]
                        for i in range(3)], 1)


def _covers(S, px, py):
    """Exact coverage with the top-left rule, and the edge functions."""
    E = _edges(S, px, py)
    s = torch.sign(E.sum(1, keepdim=True))
    X, Y = S[..., 0], S[..., 1]
    ga = torch.stack([Y[:, (i + 1) % 3] - Y[:, (i + 2) % 3] for i in range(3)], 1) * s
    gb = torch.stack([X[:, (i + 2) % 3] - X[:, (i + 1) % 3] for i in range(3)], 1) * s
    top_left = (ga > 0) | ((ga == 0) & (gb > 0))
    e = E * s
    return (((e > 0) | ((e == 0) & top_left)).all(1)) & (s[:, 0] != 0), E


def _raster64(scr, tris, H, W):
    """Index image by exact integer coverage and the largest interpolated 1/Z, ties to the lower id."""
    snap = torch.round(256.0 * scr[:, :2]).long()
    S = snap[tris]
    zeta = scr[:, 2][tris]
    lo, hi = S.amin(1), S.amax(1)
    x0, y0 = torch.div(lo + 127, 256, rounding_mode="floor").clamp(min=0).unbind(1)
    x1 = torch.div(hi[:, 0] - 128, 256, rounding_mode="floor").clamp(max=W - 1)
    y1 = torch.div(hi[:, 1] - 128, 256, rounding_mode="floor").clamp(max=H - 1)
    bw, bh = (x1 - x0 + 1).clamp(min=0), (y1 - y0 + 1).clamp(min=0)
    cnt = bw * bh
    zbuf = torch.zeros(H * W, dtype=torch.float64, device=DEV)
    ids = torch.full((H * W,), len(tris), dtype=torch.long, device=DEV)
    order = torch.nonzero(cnt > 0).flatten()
    total = torch.cumsum(cnt[order], 0)
    chunks, start = [], 0
    step = 8_000_000
    ends = [] if not len(order) else list(range(step, int(total[-1]) + step, step))
    for e in ends:
        stop = int(torch.searchsorted(total, torch.tensor(e, device=DEV), right=True))
        stop = max(stop, min(start + 1, len(order)))
        if stop > start:
            chunks.append(order[start:stop])
            start = stop
    if start < len(order):
        chunks.append(order[start:])

    def fragments(tri):
        c = cnt[tri]
        t = torch.repeat_interleave(tri, c)
        k = torch.arange(len(t), device=DEV) - torch.repeat_interleave(torch.cumsum(c, 0) - c, c)
        x, y = x0[t] + k % bw[t], y0[t] + k // bw[t]
        ok, E = _covers(S[t], 256 * x + 128, 256 * y + 128)
        t, p, E = t[ok], (y * W + x)[ok], E[ok].double()
        return t, p, (E * zeta[t]).sum(1) / E.sum(1)

    for tri in chunks:
        t, p, z = fragments(tri)
        zbuf.scatter_reduce_(0, p, z, "amax")
    for tri in chunks:
        t, p, z = fragments(tri)
        win = z == zbuf[p]
        ids.scatter_reduce_(0, p[win], t[win], "amin")
    ids[ids == len(tris)] = -1
    return ids, snap


def _bary64(v, px, py):
    """Screen barycentrics [m,3] of the pixel centres with respect to triangles v [m,3,3] (x, y, 1/Z)."""
    dx, dy = v[..., 0] - px[:, None], v[..., 1] - py[:, None]
    e = torch.stack([dx[:, (i + 1) % 3] * dy[:, (i + 2) % 3] - dy[:, (i + 1) % 3] * dx[:, (i + 2) % 3]
                     for i in range(3)], 1)
    return e / e.sum(1, keepdim=True)


def _bilinear64(tex, uv):
    """Texture [h,w,4] at uv [m,2]: u wraps, v clamps (a clamped v has no derivative)."""
    h, w = tex.shape[:2]
    fx, fy = uv[:, 0] * w - 0.5, uv[:, 1] * h - 0.5
    i, j = torch.floor(fx.detach()), torch.floor(fy.detach())
    a = fx - i
    low, high = j < 0, fy.detach() >= h - 1
    b = torch.where(low | high, torch.zeros_like(fy), fy - j)
    j0 = torch.where(low, torch.zeros_like(j), torch.where(high, torch.full_like(j, h - 1), j)).long()
    j1 = torch.where(low | high, j0, j0 + 1)
    i0 = i.long() % w
    i1 = (i0 + 1) % w
    tex = tex.double()
    top = tex[j0, i0] + a[:, None] * (tex[j0, i1] - tex[j0, i0])
    bot = tex[j1, i0] + a[:, None] * (tex[j1, i1] - tex[j1, i0])
    return top + b[:, None] * (bot - top)


def _shade64(v, lam, attr, tex, sh):
    """Shaded channels [m,C] of fragments with screen barycentrics lam on triangles v, vertex attributes attr."""
    zeta = v[..., 2]
    s = (lam * zeta).sum(1, keepdim=True)
    b = lam * zeta / s
    val = (b[:, :, None] * attr).sum(1)
    if "uv_offset" in sh:
        val = _bilinear64(tex, val)[:, :3]
    out = [val]
    if "mask_ch" in sh:
        out.append(torch.ones_like(s))
    if "depth_ch" in sh:
        out.append(1.0 / s)
    return torch.cat(out, 1)


def _pairs64(ids, snap, scr, tris, H, W):
    """Every scattering (fragment p, neighbour q): pixels, pair axis, the sign of Eq. 11 and the direction (x, y, 1/Z)
    that dL/dp is multiplied by (unit axis for an overhang, Eq. 12 at an intersection)."""
    img = ids.view(H, W)
    lin = torch.arange(H * W, device=DEV).view(H, W)
    out = []
    for axis, a, b in ((0, (slice(None), slice(0, -1)), (slice(None), slice(1, None))),
                       (1, (slice(0, -1), slice(None)), (slice(1, None), slice(None)))):
        for p_is_a in (True, False):
            P, Q = (a, b) if p_is_a else (b, a)
            tp, tq, p, q = img[P].flatten(), img[Q].flatten(), lin[P].flatten(), lin[Q].flatten()
            keep = (tp >= 0) & (tp != tq)
            tp, tq, p, q = tp[keep], tq[keep], p[keep], q[keep]
            fg = tq >= 0
            tqs = tq.clamp(min=0)
            at = [256 * (p % W) + 128, 256 * torch.div(p, W, rounding_mode="floor") + 128]
            aq = [256 * (q % W) + 128, 256 * torch.div(q, W, rounding_mode="floor") + 128]
            over = ~fg | _covers(snap[tris[tqs]], *at)[0]
            inter = fg & over & _covers(snap[tris[tp]], *aq)[0]
            p, q, tp, tqs, inter = p[over], q[over], tp[over], tqs[over], inter[over]
            d = torch.zeros((len(p), 3), dtype=torch.float64, device=DEV)
            d[:, axis] = 1.0
            if bool(inter.any()):
                vp, vq = scr[tris[tp[inter]]], scr[tris[tqs[inter]]]
                Nv = torch.linalg.cross(vp[:, 1] - vp[:, 0], vp[:, 2] - vp[:, 0])
                Nf = torch.linalg.cross(vq[:, 1] - vq[:, 0], vq[:, 2] - vq[:, 0])
                den = Nf[:, axis] * Nv[:, 2] - Nf[:, 2] * Nv[:, axis]
                mag = torch.sqrt((Nv[:, axis] ** 2 + Nv[:, 2] ** 2) * (Nf[:, axis] ** 2 + Nf[:, 2] ** 2))
                k = torch.where(den.abs() > 1e-12 * mag, -Nf[:, 2] / den, torch.zeros_like(den))
                di = torch.zeros((len(k), 3), dtype=torch.float64, device=DEV)
                di[:, axis], di[:, 2] = k * Nv[:, axis], k * Nv[:, 2]
                d[inter] = di
            out.append((p, q, 1.0 if p_is_a else -1.0, d))
    return out


def _view64(verts, attr, tris, cam, H, W, sh, tex, upstream=None, tangent=None, target=None):
    """One view: (image [H W, C], derivative image or None); with `upstream` [H W, C] or `target` (squared error),
    gradients are added to verts.grad and attr.grad."""
    tris = tris.long()
    scr = _project64(verts, cam)
    fixed = scr.detach()
    ids, snap = _raster64(fixed, tris, H, W)
    px = torch.nonzero(ids >= 0).flatten()
    cx, cy = (px % W).double() + 0.5, torch.div(px, W, rounding_mode="floor").double() + 0.5
    tri = tris[ids[px]]
    bg = torch.tensor(sh["bg"], dtype=torch.float64, device=DEV)

    def shaded(pos, at):
        v = pos[tri]
        return _shade64(v, _bary64(v, cx, cy), at[tri], tex, sh)

    val = shaded(scr, attr)
    image = bg.repeat(H * W, 1)
    image[px] = val.detach()
    if target is not None:
        upstream = 2.0 * (image - target)
    deriv = None
    lam = None
    if upstream is not None or tangent is not None:
        lam = torch.zeros((H * W, 3), dtype=torch.float64, device=DEV)
        lam[px] = _bary64(fixed[tri], cx, cy)
        pairs = _pairs64(ids, snap, fixed, tris, H, W)
    if upstream is not None:
        g = upstream.double()
        total = (val * g[px]).sum()
        for p, q, sign, d in pairs:
            dl = 0.5 * ((g[p] + g[q]) * (image[p] - image[q])).sum(1) * sign
            w = (dl[:, None] * d)[:, None, :] * lam[p][:, :, None]
            total = total + (scr[tris[ids[p]]] * w).sum()
        total.backward()
    if tangent is not None:
        with torch.no_grad():
            tv = torch.func.jvp(lambda x: _project64(x, cam), (verts.detach(),), (tangent.double(),))[1]
            deriv = torch.zeros_like(image)
            deriv[px] = torch.func.jvp(lambda x: shaded(x, attr.detach()), (fixed,), (tv,))[1]
            for p, q, sign, d in pairs:
                move = (lam[p][:, :, None] * tv[tris[ids[p]]]).sum(1)
                step = 0.5 * sign * (image[p] - image[q]) * (move * d).sum(1, keepdim=True)
                deriv.index_add_(0, p, step)
                deriv.index_add_(0, q, step)
    return image, deriv


def _solve64(tris, V, lam, b):
    """(I + lam L) x = b by conjugate gradients in 64 bits to rounding level."""
    t = tris.long()
    e = torch.cat([t[:, [0, 1]], t[:, [1, 2]], t[:, [2, 0]]])
    e = torch.unique(torch.cat([e, e.flip(1)]), dim=0)
    deg = torch.bincount(e[:, 0], minlength=V).double()[:, None]

    def M(x):
        return x + lam * (deg * x - torch.zeros_like(x).index_add_(0, e[:, 0], x[e[:, 1]]))

    b = b.double()
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), (r * r).sum()
    stop = 1e-28 * rr
    for _ in range(600):
        if rr <= stop:
            break
        q = M(p)
        a = rr / (p * q).sum()
        x, r = x + a * p, r - a * q
        new = (r * r).sum()
        p, rr = r + (new / rr) * p, new
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        v, t = _mesh(case["mesh"], case["n"], seed)
        return dict(x=_solve64(t, len(v), case["lam"], torch.randn(v.shape, generator=_gen(seed + 5), device=DEV)))
    if kind == "fit":
        items, sh = _fit_items(case, seed), SHADINGS["normals_mask"]
        rng, images, grads = np.random.default_rng(seed), [], []
        noise = rng.normal(0.0, FIT_SIGMA, (sum(len(it.verts) for it in items), 3)).astype(np.float32)
        row = 0
        for it in items:
            true, tris = torch.from_numpy(it.verts).to(DEV), torch.from_numpy(it.tris).to(DEV)
            x = (true + torch.from_numpy(noise[row:row + len(true)]).to(DEV)).double().requires_grad_(True)
            row += len(true)
            with torch.no_grad():
                target = _view64(true.double(), _normals(true.double(), tris), tris, it.cams[0], it.H, it.W, sh, None)[0]
            images.append(_view64(x, _normals(x, tris), tris, it.cams[0], it.H, it.W, sh, None, target=target)[0])
            grads.append(x.grad)
        return dict(image=torch.cat(images), index=None, grad_verts=torch.cat(grads))
    verts, tris, _, attr, tex, cams = _scene(case, seed)
    sh, n, H, W = SHADINGS[case["shade"]], case["views"], case["H"], case["W"]
    g = None if kind == "jvp" else _upstream(case, sh["C"], seed).view(n, H * W, -1)
    tangent = _tangent(verts, seed) if kind == "jvp" else None
    v, a = verts.double().requires_grad_(True), attr.double().requires_grad_(True)
    images = torch.empty((n, H * W, sh["C"]), dtype=torch.float64, device=DEV)
    for k in range(n):
        image, deriv = _view64(v, a, tris, cams[k], H, W, sh, tex, None if g is None else g[k], tangent)
        images[k] = image if deriv is None else deriv
    if kind == "jvp":
        return dict(derivative=images.view(n, H, W, -1))
    if kind == "autograd":
        return dict(image=images.view(n, H, W, -1), grad_verts=v.grad, grad_attr=a.grad)
    return dict(image=images.view(-1, sh["C"]) if kind == "graph" else images.view(n, H, W, -1), index=None,
                grad_verts=v.grad)
