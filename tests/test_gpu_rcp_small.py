"""rcp_nr at the inputs that its estimate takes for zero or that have no reciprocal: every denormal, zeros, infinities and NaN
give the correctly rounded reciprocal to one unit in the last place, and an image drawn from 1e38 away has its depth."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_rcp_nr_of_small_values(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "rcp_small_check")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "-I", os.path.join(ROOT, "include"), "-o", exe,
                    os.path.join(ROOT, "tests", "gpu_src", "rcp_small_check.cu")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    _, worst = (int(v) for v in r.stdout.split())
    assert worst <= 1, f"largest difference {worst} ulp"


def test_far_away():
    import torch

    from paper_2405_02508_gb300 import binding as B
    from paper_2405_02508_gb300.render import Renderer
    from paper_2405_02508_gb300.scenes import Shading

    H = W = 16
    z = 1.5e38  # 1 / z is denormal
    scr = torch.tensor([[[1.0, 1.0, 1 / z], [15.0, 1.0, 1 / z], [1.0, 15.0, 1 / z]]], dtype=torch.float64, device="cuda")
    r = Renderer(torch.tensor([[0, 1, 2]]), 3, 1, H, W, Shading(n_main=1, C=2, depth_ch=1, bg=[0.0, 0.0]), 1)
    r.project_screen(scr)
    r.rasterize()
    r.shade(torch.full((3, 1), 0.5, device="cuda"), None)
    drawn = (r.index[0] == 0).cpu().numpy()
    image = r.image[0].cpu().numpy()
    assert drawn.sum() > 50
    # a denormal of this size has 22 bits
    np.testing.assert_allclose(image[drawn, 1], z, rtol=2.0 ** -20)
    np.testing.assert_allclose(image[drawn, 0], 0.5, rtol=2.0 ** -20)
