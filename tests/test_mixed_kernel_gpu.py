"""Large XTS and ECB encryptions, which table warps and bitsliced warps share,
bit-exact against the CPU oracle: at the size from which bitsliced warps take
part (1,300 chunks of 512 bytes an SM with AES-256-XTS, 1,400 with AES-128) and
one unit below it, with units of exactly one chunk, units that straddle chunks
and spans, long units, ragged ends, in and out of place."""
import numpy as np
import pytest

import oracle
import workloads as w
from conftest import to_dev, to_np

pytestmark = pytest.mark.gpu


def sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("bits,du,units", [
    (128, 512, lambda s: 1400 * s),              # at the line: a unit is a chunk, 32 units a span
    (128, 512, lambda s: 1400 * s - 1),          # below it
    (256, 528, lambda s: 1300 * s * 32 // 33 + 2),  # 33 blocks: 32 units touch a span, uneven shares
    (256, 4096, lambda s: 163 * s + 1),
    (256, 4112, lambda s: 165 * s),              # 257 blocks, the last chunk is partial
    (128, 65536, lambda s: 11 * s + 3),          # a unit is four spans
    (256, 4096, lambda s: 326 * s + 5),          # two spans a warp
])
def test_mixed_xts(ctx, bits, du, units):
    n = units(sms())
    key = w.xts_key(51, bits)
    first = 2**40 + 13
    data = w.seeded_bytes(51 + du, w.STREAM_DATA, du * n)
    ref = oracle.xts(key, 0, data, du, first)
    kh = ctx.setkey(key, True)
    try:
        for in_place in (False, True):
            src = to_dev(data)
            dst = src if in_place else src.new_empty(src.shape)
            ctx.xts_crypt(kh, 0, src, dst, du, first)
            assert np.array_equal(to_np(dst), ref), (bits, du, n, in_place)
    finally:
        ctx.delkey(kh)


@pytest.mark.parametrize("bits", [128, 192, 256])
def test_mixed_ecb(ctx, bits):
    n = 16 * (sms() * 32 * 1400 + 37)  # over the line, with a partial last chunk
    key = w.single_key(52, bits)
    data = w.seeded_bytes(52 + bits, w.STREAM_DATA, n)
    ref = oracle.ecb(key, 0, data)
    kh = ctx.setkey(key, False)
    try:
        for in_place in (False, True):
            src = to_dev(data)
            dst = src if in_place else src.new_empty(src.shape)
            ctx.ecb_crypt(kh, 0, src, dst)
            assert np.array_equal(to_np(dst), ref), (bits, in_place)
    finally:
        ctx.delkey(kh)
