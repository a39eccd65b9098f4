"""Which form a bulk call takes, decided by the library from its sizes, on the
CPU through a small C++ harness (tests/bulk_rules_check.cc): every form gives
the same bytes, so the tests of results cannot tell which one ran."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SMS = 152


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    cxx = shutil.which("g++")
    cuda_inc = "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are not available")
    exe = str(tmp_path_factory.mktemp("rules") / "bulk_rules_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_1305_3345_gb300", "csrc"), "-I", cuda_inc,
                    os.path.join(HERE, "bulk_rules_check.cc"), "-o", exe], check=True)

    def run(kind, *args):
        line = " ".join(map(str, (kind, *args))) + "\n"
        return int(subprocess.run([exe], input=line, capture_output=True, text=True, check=True).stdout)
    return run


@pytest.mark.parametrize("bpp", [1, 8, 256, 257, 4096])
def test_cbc_encryption_of_device_pages(ask, bpp):
    most = 192 if bpp % 8 == 0 else 240
    for nr in (10, 12, 14):
        assert ask("e", 1, bpp, nr, SMS, 0) == 4
        assert ask("e", 32 * SMS, bpp, nr, SMS, 0) == 4
        assert ask("e", 32 * SMS + 1, bpp, nr, SMS, 0) == 2
        assert ask("e", most * SMS, bpp, nr, SMS, 0) == 2
        assert ask("e", most * SMS + 1, bpp, nr, SMS, 0) == 1


@pytest.mark.parametrize("nr,few", [(10, 32), (12, 128), (14, 256)])
def test_cbc_encryption_over_the_link_moves_whole_lines(ask, nr, few):
    """Pages in whole 128-byte lines are staged, but for a few pages; shared
    lanes would move 16 bytes a page at a time."""
    for bpp in (8, 32, 256, 4096):
        assert ask("e", few, bpp, nr, SMS, 1) == 4
        for n in (few + 1, 4096, 32 * SMS + 1, 192 * SMS):
            assert ask("e", n, bpp, nr, SMS, 1) == 1
    # what cannot be staged is as on the device
    assert ask("e", 32 * SMS, 257, nr, SMS, 1) == 4
    assert ask("e", 240 * SMS, 257, nr, SMS, 1) == 2


def test_split_chains_leave_sms_to_other_streams(ask):
    """At least one CTA, never more than SMs or 16 warps to one, two warps an SM
    while that takes an eighth of the SMs, at most three further on."""
    last = 0
    for teams in list(range(1, 400)) + [1216, 1824, 1825, 2432]:
        n = ask("s", teams, SMS)
        assert 1 <= n <= SMS and n >= last and n * 16 >= teams
        last = n
        if teams <= 2 * (SMS // 8):
            assert n == (teams + 1) // 2
        elif teams <= 3 * SMS:
            assert n == max(SMS // 8, (teams + 2) // 3)
        else:
            assert n == SMS
    assert ask("s", 5, 1) == 1 and ask("s", 5, 7) <= 2


def test_sms_for_pages_over_the_link(ask):
    """A quarter of the SMs for short calls, three quarters for long ones, all
    for units under 512 bytes."""
    mib = 1 << 20
    for unit, most in ((32, 48), (64, 48), (128, 96), (256, 96), (1 << 20, 96)):
        assert ask("l", SMS, unit, 16) == ask("l", SMS, unit, most * mib) == 38
        assert ask("l", SMS, unit, most * mib + 1) == ask("l", SMS, unit, 1024 * mib) == 114
        assert ask("l", 1, unit, mib) == ask("l", 1, unit, 1024 * mib) == 1
    assert ask("l", SMS, 31, mib) == ask("l", SMS, 1, 1024 * mib) == SMS


def test_sms_for_cbc_decryption(ask):
    mib = 1 << 20
    for bytes_ in (4096, 4 * mib, 1024 * mib):
        assert ask("d", SMS, 256, bytes_, 0) == SMS
    assert ask("d", SMS, 256, 2 * mib - 4096, 1) == SMS
    assert ask("d", SMS, 256, 2 * mib, 1) == ask("d", SMS, 32, 48 * mib, 1) == 38
    assert ask("d", SMS, 32, 49 * mib, 1) == ask("d", SMS, 256, 97 * mib, 1) == 114
    assert ask("d", SMS, 16, 64 * mib, 1) == SMS


# name in bench.py, name in test_mixed_kernel_gpu.py: rounds, direction, tweak
MIXED = {("aes256_xts_enc", "ENC256"): (14, 0, 1), ("aes128_xts_enc", "ENC128"): (10, 0, 1),
         ("aes256_xts_dec", "DEC256"): (14, 1, 1), ("aes128_xts_dec", "DEC128"): (10, 1, 1),
         ("aes128_ecb_enc", None): (10, 0, 0), ("aes128_cbc_dec", "PLAIN"): (10, 1, 0)}


def test_bitsliced_warps_take_part_from_where_the_bench_and_the_tests_say(ask):
    """The bench scales its lookup bound by the share of the blocks that is
    looked up, and the tests of the mixed kernels go to their lines: both in
    chunks a CTA, which the library's rule must agree with."""
    import bench
    import test_mixed_kernel_gpu as gpu
    assert set(bench.CHUNKS_PER_SPAN) == {b for b, _ in MIXED}
    for (b, g), (nr, dir, tweak) in MIXED.items():
        line = bench.CHUNKS_PER_SPAN[b]
        assert g is None or getattr(gpu, g) == line
        for unit in (32, 256, 1 << 20):
            assert ask("m", line - 1, nr, dir, tweak, unit, 0) == 0
            assert ask("m", line, nr, dir, tweak, unit, 0) == 1
            assert ask("m", 10 * line + 7, nr, dir, tweak, unit, 0) == 10
        assert ask("m", 10 * line, nr, dir, tweak, 31, 0) == 0      # units under 512 bytes
        assert ask("m", 10 * line, nr, dir, tweak, 256, 1) == 0     # pages over the link
    # the spans never exceed what a CTA has: four warps, 32 chunks a span
    for chunks in (1200, 5000, 13797, 10 ** 6):
        for nr, dir, tweak in [*MIXED.values(), (12, 0, 0), (12, 1, 0), (14, 0, 0), (14, 1, 0)]:
            assert 128 * ask("m", chunks, nr, dir, tweak, 256, 0) < chunks
    assert ask("m", 10 ** 6, 12, 0, 1, 256, 0) == 0                 # there is no XTS-AES-192
    for nr in (10, 12, 14):                                         # every plain size the GPU tests run
        for dir in (0, 1):
            assert ask("m", gpu.PLAIN, nr, dir, 0, 32, 0) >= 1
