"""How the bulk kernels split a buffer over CTAs, warps and lanes, at the sizes
where the split changes, bit-exact against the CPU oracle: XTS with tweaks
formed by the whole CTA (units of at least 512 B) or by each warp (smaller
units), one phase or several; XTS units that end in ciphertext stealing, in
phases of one unit per thread and at every alignment; CBC decryption out of
place (chunks) and in place (pages); CBC encryption with one, two or four lanes
per page."""
import numpy as np
import pytest

import oracle
import workloads as w
from conftest import to_dev, to_np

pytestmark = pytest.mark.gpu


def sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def run_xts(ctx, key, dir, data, du, first, in_place):
    kh = ctx.setkey(key, True)
    try:
        src = to_dev(data)
        dst = src if in_place else src.new_empty(src.shape)
        ctx.xts_crypt(kh, dir, src, dst, du, first)
        return to_np(dst)
    finally:
        ctx.delkey(kh)


@pytest.mark.parametrize("dir", [0, 1])
@pytest.mark.parametrize("du,units", [
    (512, lambda s: s * 1024 + 3 * s + 1),   # a phase holds 1,024 of them: two phases a CTA, uneven shares
    (528, lambda s: s * 1024 + 2 * s + 5),   # 33 blocks: units straddle chunks and phases
    (4096, lambda s: 1),                     # one CTA, eight chunks
    (4096, lambda s: s // 2 + 1),            # four chunks a CTA: the last grid below one CTA per SM
    (496, lambda s: 9 * s + 1),              # 31 blocks: formed by each warp, several phases a warp
    (16, lambda s: 40 * s + 7),              # every block a unit: one chunk a phase
])
def test_xts_phases(ctx, dir, du, units):
    n = units(sms())
    key = w.xts_key(31, 256 if du != 512 else 128)
    first = 2**40 + 11
    data = w.seeded_bytes(31 + du, w.STREAM_DATA, du * n)
    ref = oracle.xts(key, dir, data, du, first)
    for in_place in (False, True):
        assert np.array_equal(run_xts(ctx, key, dir, data, du, first, in_place), ref), (du, n, in_place)


@pytest.mark.parametrize("page,npages", [
    (4096, lambda s: 1),
    (4096, lambda s: s + 1),                 # in place: two pages on one CTA
    (4096, lambda s: 4 * s + 3),             # about one chunk a warp
    (512, lambda s: 32 * s + 7),             # a page is a chunk
    (496, lambda s: 33 * s + 2),             # pages straddle chunks, warps and CTAs
    (16, lambda s: 128 * s + 5),             # every block starts a page
    (8 * 4096 + 48, lambda s: 3),            # long pages over many warps
])
def test_cbc_decrypt_split(ctx, page, npages):
    n = npages(sms())
    key = w.single_key(32, 192)
    data = w.seeded_bytes(32 + page, w.STREAM_DATA, page * n)
    ivs = w.page_ivs(32 + page, n)
    ref = oracle.cbc(key, 1, data, page, ivs)
    kh = ctx.setkey(key, False)
    try:
        iv = to_dev(np.ascontiguousarray(ivs).reshape(-1))
        for in_place in (False, True):
            src = to_dev(data)
            dst = src if in_place else src.new_empty(src.shape)
            ctx.cbc_decrypt(kh, src, dst, page, iv)
            assert np.array_equal(to_np(dst), ref), (page, n, in_place)
    finally:
        ctx.delkey(kh)


@pytest.mark.parametrize("page,npages", [
    (4096, lambda s: 1),
    (48, lambda s: 32 * s),                  # four lanes a page: the largest call
    (16, lambda s: 32 * s + 1),              # two lanes a page: the smallest, ragged team
    (128, lambda s: 192 * s),                # two lanes: the largest of pages that can be staged
    (128, lambda s: 192 * s + 1),            # one lane
    (48, lambda s: 240 * s + 9),             # one lane, pages that cannot be staged
    (80, lambda s: 240 * s - 3),             # two lanes: several waves of warps
])
@pytest.mark.parametrize("bits", [128, 192, 256])
def test_cbc_encrypt_lanes(ctx, bits, page, npages):
    n = npages(sms())
    key = w.single_key(33, bits)
    data = w.seeded_bytes(33 + page, w.STREAM_DATA, page * n)
    ivs = w.page_ivs(33 + page, n)
    ref = oracle.cbc(key, 0, data, page, ivs)
    kh = ctx.setkey(key, False)
    try:
        iv = to_dev(np.ascontiguousarray(ivs).reshape(-1))
        for in_place in (False, True):
            src = to_dev(data)
            dst = src if in_place else src.new_empty(src.shape)
            ctx.cbc_encrypt_pages(kh, src, dst, page, iv)
            assert np.array_equal(to_np(dst), ref), (bits, page, n, in_place)
    finally:
        ctx.delkey(kh)


@pytest.mark.parametrize("dir", [0, 1])
@pytest.mark.parametrize("du,units", [
    (24, lambda s: 768 * s + 2 * s + 1),     # 8-byte accesses, two phases a CTA
    (19, lambda s: 768 * s + 5),             # byte alignment, one block a unit
    (18, lambda s: 5 * s),                   # 2-byte alignment
    (20, lambda s: 1),                       # one unit, the whole buffer 20 bytes
    (520, lambda s: 4 * s + 1),              # 32 blocks and a half: a chunk a unit
    (1037, lambda s: 97),                    # 64 blocks and 13 bytes, fewer units than SMs
    (70002, lambda s: 3),                    # long units
])
def test_xts_stealing_phases(ctx, dir, du, units):
    n = units(sms())
    key = w.xts_key(34, 128 if du % 2 else 256)
    first = 2**33 + 5
    data = w.seeded_bytes(34 + du, w.STREAM_DATA, du * n)
    ref = oracle.xts(key, dir, data, du, first)
    for in_place in (False, True):
        assert np.array_equal(run_xts(ctx, key, dir, data, du, first, in_place), ref), (du, n, in_place)
