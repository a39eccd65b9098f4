"""How batched and served requests are cut and ordered, on the CPU through a
small C++ harness built against the library's own header (tests/plan_check.cc)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SMS = 152
WORKERS = SMS * 16 - 1
MIB = 1 << 20


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    cxx = shutil.which("g++")
    cuda_inc = "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are not available")
    exe = str(tmp_path_factory.mktemp("plan") / "plan_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_1305_3345_gb300", "csrc"), "-I", cuda_inc,
                    os.path.join(HERE, "plan_check.cc"), "-o", exe], check=True)

    def run(*words):
        text = " ".join(map(str, words)) + "\n"
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [[int(x) for x in line.split()] for line in out.splitlines()]
    return run


def test_burst_tiles(ask):
    """A burst on device pages takes larger tiles, one on host pages the default,
    unless the request would then have more tiles than the ring takes."""
    def tile(burst, nblocks=256, host=0, most=1 << 22):
        return ask("b", 2, nblocks, burst, WORKERS, host, most)[0][0]
    assert tile(4096) == tile(2 * 4096 * WORKERS - 1) == 2
    assert tile(2 * 4096 * WORKERS) == 4
    assert tile(1 << 40) == 64
    for burst in (4096, 24 * MIB, 160 * MIB, 1 << 40):
        assert tile(burst, host=1) == 2
    assert tile(1 << 40, nblocks=2 * 32 * 1000, host=1, most=1000) == 2
    assert tile(1 << 40, nblocks=2 * 32 * 1000 + 1, host=1, most=1000) == 64
