"""The tweak of a block far inside a long data unit: T * x^j in GF(2^128) by
square and multiply (csrc/gf128_jump.cuh), against carry-less integer
arithmetic, on the CPU through a small C++ harness (tests/gf128_check.cc)."""
import os
import random
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++")
    cuda_inc = "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are not available")
    exe = str(tmp_path_factory.mktemp("gf128") / "gf128_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_1305_3345_gb300", "csrc"), "-I", cuda_inc,
                    os.path.join(HERE, "gf128_check.cc"), "-o", exe], check=True)
    return exe


def times(a, b):
    p = 0
    while b:
        if b & 1:
            p ^= a
        b >>= 1
        a <<= 1
        if a >> 128:
            a ^= (1 << 128) | 0x87
    return p


def power_of_x(j):
    r = 1
    for bit in bin(j)[2:]:
        r = times(r, r)
        if bit == "1":
            r = times(r, 2)
    return r


def test_jump_equals_integer_arithmetic(harness):
    rng = random.Random(3)
    js = [64, 127, 128, 129, 255, 256, 8191, 8192, 2**20 - 1, 2**20, 2**31, 2**32 - 1]
    js += [rng.randrange(64, 2 ** rng.randrange(7, 33)) for _ in range(300)]
    ts = [1, 1 << 127, (1 << 128) - 1] + [rng.getrandbits(128) for _ in range(len(js))]
    cases = [(t, j) for j in js[:12] for t in ts[:6]] + list(zip(ts[6:], js[12:]))
    text = "".join(" ".join(f"{t >> 32 * i & 0xffffffff:x}" for i in range(4)) + f" {j}\n" for t, j in cases)
    out = subprocess.run([harness], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    for (t, j), line in zip(cases, out):
        got = sum(int(w, 16) << 32 * i for i, w in enumerate(line.split()))
        assert got == times(t, power_of_x(j)), (hex(t), j)
