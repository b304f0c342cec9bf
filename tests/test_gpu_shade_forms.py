"""The layout forms of the shading (three textured channels, three interpolated ones) against the generic form: the same
scene in a layout that only the generic form takes gives the same image bit for bit and the same gradients, also at texture
sizes of one texel, clamped and wrapped coordinates, and coordinates that are out of range or not finite."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2405_02508_gb300 import scenes
from paper_2405_02508_gb300.scenes import Shading

pytestmark = pytest.mark.gpu


def _run(sh, attr, tex, g, batched):
    """(image, grad_vpix, grad_attr) of two views of a sphere."""
    import torch

    from paper_2405_02508_gb300 import binding as B
    from paper_2405_02508_gb300.batch import BatchRenderer
    from paper_2405_02508_gb300.render import Renderer

    H, W = 75, 101
    P, F = scenes.octasphere(12)
    cams = scenes.cameras_on_sphere(2, 3.0, H, W, 3)
    verts = torch.from_numpy(P.astype(np.float32)).cuda()
    a = torch.from_numpy(attr).cuda()
    t = None if tex is None else torch.from_numpy(tex).cuda()
    ga = torch.zeros_like(a)
    if batched:
        br = BatchRenderer([(P, F.astype(np.int32))], [(0, k, H, W) for k in range(2)], cams, sh, attr.shape[1], t, tile=32)
        br.prepare(verts, a, t)
        br.backward(torch.from_numpy(g).cuda().view(-1, sh.C), a, t, grad_attr=ga)
        br.check()
        return br.image.cpu().numpy().reshape(2, H, W, -1), br.grad_vpix.cpu().numpy(), ga.cpu().numpy()
    r = Renderer(torch.from_numpy(F.astype(np.int32)), len(P), 2, H, W, sh, attr.shape[1], None if t is None else t.shape)
    c = B.cameras_tensor(cams)
    r.forward(verts, c, a, t)
    r.backward(torch.from_numpy(g).cuda(), c, a, t, grad_attr=ga)
    r.check_status()
    return r.image.cpu().numpy(), r.grad_vpix.cpu().numpy(), ga.cpu().numpy()


def _same(x, y, a, b):
    """Sums of the same FP32 terms in another order: within 2^-24 times the number of terms (at most 512 a tile) of the
    largest sum."""
    np.testing.assert_allclose(x, y, rtol=512 * 2.0 ** -24, atol=512 * 2.0 ** -24 * max(np.abs(y).max(), 1e-30))
    np.testing.assert_allclose(a, b, rtol=512 * 2.0 ** -24, atol=512 * 2.0 ** -24 * max(np.abs(b).max(), 1e-30))


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("size", [(1, 1), (1, 5), (7, 1), (2, 3), (64, 64)])
@pytest.mark.parametrize("values", ["plain", "wild"])
def test_textured(batched, size, values):
    P, _ = scenes.octasphere(12)
    rng = np.random.default_rng(5)
    uv = scenes.equirect_uv(P).astype(np.float32)
    if values == "wild":
        uv = (uv * 6 - 3).astype(np.float32)
        uv[::11] = [2000.0, 0.5]
        uv[5::17] = [0.5, np.inf]
        uv[7::19] = [np.nan, 0.2]
    tex = rng.uniform(0, 1, (*size, 4)).astype(np.float32)
    wide = np.concatenate([uv, rng.uniform(0, 1, (len(uv), 1)).astype(np.float32)], axis=1)  # three floats a vertex: generic
    sh = Shading(n_main=3, C=5, uv_offset=0, mask_ch=3, depth_ch=4, bg=[0.1, 0.2, 0.3, 0.0, 0.0])
    g = rng.standard_normal((2, 75, 101, 5)).astype(np.float32)
    fi, fv, fa = _run(sh, uv, tex, g, batched)
    gi, gv, gat = _run(sh, wide, tex, g, batched)
    np.testing.assert_array_equal(fi, gi)
    if values == "plain":
        _same(fv, gv, fa, gat[:, :2])
    else:  # not finite where a triangle has such a coordinate, in both
        np.testing.assert_array_equal(np.isfinite(fv), np.isfinite(gv))


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("extra", [0, 2])
def test_interpolated(batched, extra):
    P, _ = scenes.octasphere(12)
    rng = np.random.default_rng(6)
    attr = rng.uniform(-1, 1, (len(P), 4 + extra)).astype(np.float32)
    g = rng.standard_normal((2, 75, 101, 5)).astype(np.float32)
    g[..., 3] = 0.0
    four = Shading(n_main=4, C=5, mask_ch=4, bg=[0.1, 0.2, 0.3, 0.4, 0.0])  # four channels: generic
    three = Shading(n_main=3, C=4, mask_ch=3, bg=[0.1, 0.2, 0.3, 0.0])
    keep = [0, 1, 2, 4]
    gi, gv, gat = _run(four, attr, None, g, batched)
    three_attr = np.ascontiguousarray(attr[:, [0, 1, 2] + list(range(4, 4 + extra))])
    fi, fv, fa = _run(three, three_attr, None, np.ascontiguousarray(g[..., keep]), batched)
    np.testing.assert_array_equal(fi, gi[..., keep])
    _same(fv, gv, fa[:, :3], gat[:, :3])
