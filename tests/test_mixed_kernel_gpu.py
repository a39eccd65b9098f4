"""Large XTS, ECB and CBC-decryption calls, which table warps and bitsliced
warps share, bit-exact against the CPU oracle: at the size from which bitsliced
warps take part (a number of 512-byte chunks an SM that depends on the cipher)
and one unit below it, with units of exactly one chunk, units that straddle
chunks and spans, long units, ragged ends, in and out of place."""
import numpy as np
import pytest

import oracle
import workloads as w
from conftest import to_dev, to_np

pytestmark = pytest.mark.gpu


def sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


# chunks per SM from which a bitsliced warp takes a span: XTS encryption and
# decryption with either key size, ECB and CBC at most
ENC256, ENC128, DEC256, DEC128, PLAIN = 1300, 1400, 1600, 1800, 1300


@pytest.mark.parametrize("bits,dir,du,units", [
    (128, 0, 512, lambda s: ENC128 * s),              # at the line: a unit is a chunk, 32 units a span
    (128, 0, 512, lambda s: ENC128 * s - 1),          # below it
    (256, 0, 528, lambda s: ENC256 * s * 32 // 33 + 2),  # 33 blocks: 32 units touch a span, uneven shares
    (256, 0, 4112, lambda s: 165 * s),                # 257 blocks, the last chunk is partial
    (128, 0, 65536, lambda s: 11 * s + 3),            # a unit is four spans
    (256, 0, 4096, lambda s: 326 * s + 5),            # two spans a warp
    (128, 1, 512, lambda s: DEC128 * s),
    (128, 1, 512, lambda s: DEC128 * s - 1),
    (256, 1, 528, lambda s: DEC256 * s * 32 // 33 + 2),
    (256, 1, 4096, lambda s: 2 * DEC256 * s // 8 + 5),
])
def test_mixed_xts(ctx, bits, dir, du, units):
    n = units(sms())
    key = w.xts_key(51, bits)
    first = 2**40 + 13
    data = w.seeded_bytes(51 + du, w.STREAM_DATA, du * n)
    ref = oracle.xts(key, dir, data, du, first)
    kh = ctx.setkey(key, True)
    try:
        for in_place in (False, True):
            src = to_dev(data)
            dst = src if in_place else src.new_empty(src.shape)
            ctx.xts_crypt(kh, dir, src, dst, du, first)
            assert np.array_equal(to_np(dst), ref), (bits, dir, du, n, in_place)
    finally:
        ctx.delkey(kh)


@pytest.mark.parametrize("dir", [0, 1])
@pytest.mark.parametrize("bits", [128, 192, 256])
def test_mixed_ecb(ctx, bits, dir):
    n = 16 * (sms() * 32 * PLAIN + 37)  # over the line, with a partial last chunk
    key = w.single_key(52, bits)
    data = w.seeded_bytes(52 + bits, w.STREAM_DATA, n)
    ref = oracle.ecb(key, dir, data)
    kh = ctx.setkey(key, False)
    try:
        for in_place in (False, True):
            src = to_dev(data)
            dst = src if in_place else src.new_empty(src.shape)
            ctx.ecb_crypt(kh, dir, src, dst)
            assert np.array_equal(to_np(dst), ref), (bits, dir, in_place)
    finally:
        ctx.delkey(kh)


@pytest.mark.parametrize("bits,page,npages", [
    (128, 512, lambda s: PLAIN * s),                # at the line: a page is a chunk
    (192, 4096, lambda s: 2 * PLAIN * s // 8 + 7),  # two spans a warp
    (256, 4112, lambda s: PLAIN * s // 8),          # pages straddle chunks and spans
    (128, 528, lambda s: PLAIN * s),                # every lane step enters a page
    (256, 8 * 4096 + 48, lambda s: PLAIN * s // 64 + 1),
])
def test_mixed_cbc_decrypt(ctx, bits, page, npages):
    n = npages(sms())
    key = w.single_key(53, bits)
    data = w.seeded_bytes(53 + page, w.STREAM_DATA, page * n)
    ivs = w.page_ivs(53 + page, n)
    ref = oracle.cbc(key, 1, data, page, ivs)
    kh = ctx.setkey(key, False)
    try:
        iv = to_dev(np.ascontiguousarray(ivs).reshape(-1))
        for in_place in (False, True):  # in place it stays on the tables
            src = to_dev(data)
            dst = src if in_place else src.new_empty(src.shape)
            ctx.cbc_decrypt(kh, src, dst, page, iv)
            assert np.array_equal(to_np(dst), ref), (bits, page, n, in_place)
    finally:
        ctx.delkey(kh)
