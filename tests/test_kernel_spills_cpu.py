"""Registers of the batch and serving kernels: none of them may spill, which
shows in no result but in every tile's time (nvcc's own report)."""
import os
import re
import subprocess

import pytest

import paper_1305_3345_gb300.build as build


def test_batch_and_serving_kernels_do_not_spill(tmp_path):
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc is not available")
    r = subprocess.run([nvcc, *build.ARCH, *build.NVCC_FLAGS, "-Xptxas", "-v", "-I", build.INCLUDE, "-I", build.CSRC,
                        "-c", os.path.join(build.CSRC, "kgpu_unified.cu"), "-o", str(tmp_path / "u.o")],
                       capture_output=True, text=True, check=True)
    kernel, seen = None, {}
    for line in r.stderr.splitlines():
        m = re.search(r"Compiling entry function '\w*?(batch_kernelILi\d+|serve_kernelILi\d+)", line)
        if m:
            kernel = m.group(1)
        m = re.search(r"(\d+) bytes stack frame, (\d+) bytes spill stores, (\d+) bytes spill loads", line)
        if m and kernel:
            seen[kernel] = tuple(map(int, m.groups()))
            kernel = None
    assert {"batch_kernelILi512", "batch_kernelILi1024", "serve_kernelILi512"} <= set(seen), r.stderr
    assert set(seen.values()) == {(0, 0, 0)}, seen
