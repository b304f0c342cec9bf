"""The projection without 64-bit conversions: f2d and i2d on every 32-bit pattern, and snapping at its limits (ties, the
guard band, values that are not finite) against the definition in FP64, bit for bit."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_conversions_exact(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "convert_check")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "-I", os.path.join(ROOT, "include"), "-o", exe,
                    os.path.join(ROOT, "tests", "gpu_src", "convert_check.cu")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == ["0", "0"]


def test_snap_limits():
    import torch

    from paper_2405_02508_gb300 import binding as B

    edge = 2.0 ** 21  # the guard band in pixels
    rng = np.random.default_rng(0)
    xs = np.concatenate([(np.arange(-9, 10) + 0.5) / 256.0, np.nextafter(1.5 / 256.0, [0, 1]), [0.0, -0.0],
                         [edge, np.nextafter(edge, 0), np.nextafter(edge, 2 * edge), -edge, np.nextafter(-edge, 0),
                          np.nextafter(-edge, -2 * edge), 3e9, -3e9, 1e300, np.inf, -np.inf, np.nan],
                         rng.uniform(-3000, 3000, 2000), rng.uniform(-edge, edge, 2000)])
    scr = np.stack([xs, np.roll(xs, 7), np.where(np.arange(len(xs)) % 5 == 0, -0.25, 0.3 + 1e-9 * xs.clip(-1e3, 1e3))], 1)
    scr[:, 2] = np.where(np.isfinite(scr[:, 2]), scr[:, 2], 0.4)
    vpix = torch.empty((1, len(xs), 8), dtype=torch.float32, device="cuda")
    B.mer_project_screen(torch.from_numpy(scr[None].copy()).cuda(), vpix)
    rec = vpix[0].cpu().numpy()
    ints = rec.view(np.int32)
    inside = (scr[:, 2] > 0) & (np.abs(scr[:, 0]) <= edge) & (np.abs(scr[:, 1]) <= edge)
    np.testing.assert_array_equal(ints[:, 6], (scr[:, 2] > 0) * 1 + inside * 2)
    for c in range(2):
        v = scr[inside, c]
        snap = np.rint(256.0 * v)  # ties to even
        np.testing.assert_array_equal(ints[inside, c], snap.astype(np.int32))
        np.testing.assert_array_equal(rec[inside, 2 + c], (v - snap / 256.0).astype(np.float32))
        assert not ints[~inside, c].any() and not rec[~inside, 2 + c].any()
    front = scr[:, 2] > 0
    hi = scr[front, 2].astype(np.float32)
    np.testing.assert_array_equal(rec[front, 4], hi)
    np.testing.assert_array_equal(rec[front, 5], (scr[front, 2] - hi.astype(np.float64)).astype(np.float32))
