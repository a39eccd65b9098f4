"""How batched and served requests are cut and ordered, on the CPU through a
small C++ harness built against the library's own header (tests/plan_check.cc)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SMS = 152
WORKERS = SMS * 16 - 1
MIB = 1 << 20
XTS, CBC_DEC, CBC_ENC, ECB = 0, 1, 2, 3
SRC_HOST, SPLIT = 1, 8


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


def test_ctas_beyond_the_sms_do_not_run_at_once(ask):
    assert ask("r", SMS, SMS) == ask("r", 304, SMS) == ask("r", 4096, SMS) == [[SMS]]
    assert ask("r", 3, SMS) == [[3]]
    lens = [MIB] * 40  # 80 Ki chunks: 16-KiB tiles fill 2,432 warps, more CTAs change nothing
    assert ask("t", SMS, SMS, 16, 40, *lens) == ask("t", 4096, SMS, 16, 40, *lens) == [[32]]
    assert ask("t", SMS, SMS, 16, 1, 4096) == [[2]]


def plan(ask, ctas, warps, reqs):
    head, order, prefix, form = ask("p", ctas, SMS, warps, len(reqs), *(x for r in reqs for x in r))
    return head, order, prefix, list(zip(form[::2], form[1::2]))


@pytest.mark.parametrize("warps", [16, 32])
@pytest.mark.parametrize("ctas", [3, SMS, 700])
@pytest.mark.parametrize("seed", range(4))
def test_plan(ask, seed, ctas, warps):
    """CBC encryption first and smallest first, the rest after it, smallest
    first; what the header says of both; lanes per chain."""
    rng = np.random.default_rng(seed)
    reqs = []
    for _ in range(1 + 60 * seed):
        mode = int(rng.choice([XTS, CBC_DEC, CBC_ENC, ECB]))
        nb = 256 * int(rng.integers(0, 300)) if rng.integers(0, 15) else 0
        reqs.append((mode, nb, 256 if rng.integers(0, 4) else 1, 32 if mode == CBC_ENC else int(rng.choice([2, 8, 32])),
                     int(rng.integers(0, 2)) * SRC_HOST))
    (total, longs, long_warps, at_once), order, prefix, form = plan(ask, ctas, warps, reqs)
    assert at_once == min(ctas, SMS)

    def splits(r):
        return r[0] == CBC_ENC and r[1] and not (r[4] & SRC_HOST and r[2] % 8 == 0)
    chains = sum(-(-(r[1] // r[2]) // 16) for r in reqs if splits(r))
    two_lanes = warps == 16 and chains <= at_once * 16
    for r, (flags, units) in zip(reqs, form):
        assert (flags, units) == ((r[4] | SPLIT, 16) if two_lanes and splits(r) else (r[4], r[3]))

    def tiles(i):
        mode, nb, unit, _, _ = reqs[i]
        return -(-(nb // unit if mode in (CBC_DEC, CBC_ENC) else -(-nb // 32)) // form[i][1])
    assert order == sorted(range(len(reqs)), key=lambda i: (reqs[i][0] != CBC_ENC, tiles(i), i))
    assert prefix == [sum(tiles(i) for i in order[:k]) for k in range(len(order) + 1)]
    assert total == prefix[-1] and longs == sum(tiles(i) for i in range(len(reqs)) if reqs[i][0] == CBC_ENC)
    blocks = sum(r[1] for r in reqs)
    share = int(warps * 4 / 3 * sum(r[1] for r in reqs if r[0] == CBC_ENC) / blocks) + 1 if blocks else 1
    assert long_warps == min(-(-longs // at_once), share, warps)


def test_two_lanes_only_while_every_chain_runs_at_once(ask):
    """Counted in the CTAs that run at once, however many are asked for."""
    for ctas in (SMS, 304, 4096):
        for pages, split in ((16 * 16 * SMS, SPLIT), (16 * 16 * SMS + 1, 0)):
            _, _, _, form = plan(ask, ctas, 16, [(CBC_ENC, 256 * pages, 256, 32, 0)])
            assert form[0][0] == split, (ctas, pages)
