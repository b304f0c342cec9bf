"""Kernels launched so that they overlap the one before them (launch_chained): each waits in its first statement, and reads
global memory with plain loads only.  A read-only load (a const __restrict__ kernel parameter, or __ldg) may be moved ahead of the
wait, and then reads what the kernel before has not written yet.  Checked in the source."""
from __future__ import annotations

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_02508_gb300", "csrc")


def _sources():
    out = {}
    for name in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, name)).read()
        src = re.sub(r"//[^\n]*", "", src)
        out[name] = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    return out


def _kernels(src):
    """name -> (signature, body's first statement) of the __global__ functions."""
    out = {}
    for m in re.finditer(r"__global__", src):
        brace, semi = src.find("{", m.start()), src.find(";", m.start())
        if semi < brace:
            continue  # a declaration
        sig = src[m.start():brace]
        name = re.findall(r"(k_\w+)\s*\(", sig)[0]
        out[name] = (sig, src[brace + 1:src.index(";", brace)].strip())
    return out


def test_chained_kernels_wait_and_load_plainly():
    srcs = _sources()
    kernels, chained = {}, set()
    for src in srcs.values():
        kernels.update(_kernels(src))
        for call in re.finditer(r"launch_chained\(\s*(\w+)", src):
            chained.add(call.group(1))
        for alias in re.finditer(r"=\s*[^;]*?\b(k_\w+)<[^;]*;", src):  # a kernel picked before it is launched
            chained.add(alias.group(1))
    chained = {k for k in chained if k in kernels}
    assert len(chained) >= 25
    for k in sorted(chained):
        sig, first = kernels[k]
        if first.startswith("extern __shared__"):
            continue  # the solver's, launched on its own
        assert first == "after_previous()", k
        assert "__restrict__" not in sig, k
    for name, src in srcs.items():
        if "launch_chained(" in src or name.endswith(".cuh"):
            assert "__ldg(" not in src and "ld.global.nc" not in src, name
