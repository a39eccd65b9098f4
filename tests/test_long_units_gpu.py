"""XTS over long data units, whose blocks' tweaks lie far from the unit's
start: bit-exact against the CPU oracle on the tables, with bit-planes, with
ciphertext stealing and batched, and no slower for the unit's length."""
import numpy as np
import pytest

import oracle
import workloads as w
from conftest import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,dir,du,units", [
    (256, 0, 8191 * 16, 9),          # jumps end just below and at the line between the two forms
    (128, 1, 8193 * 16, 9),
    (256, 1, (1 << 20) + 16, 3),
    (128, 0, 16 << 20, 2),           # 2^20 blocks, IEEE 1619's limit
    (256, 0, (16 << 20) + 48, 2),
    (256, 0, 16 << 20, 7),           # with bit-planes
    (128, 1, (1 << 20) + 16, 144),   # with bit-planes
    (128, 0, (1 << 20) + 5, 3),      # ciphertext stealing
    (256, 1, (4 << 20) + 15, 2),
])
def test_long_units(ctx, bits, dir, du, units):
    key = w.xts_key(61, bits)
    first = 2**40 + 7
    data = w.seeded_bytes(61 + units, w.STREAM_DATA, du * units)
    ref = oracle.xts(key, dir, data, du, first)
    kh = ctx.setkey(key, True)
    try:
        for in_place in (False, True):
            src = to_dev(data)
            dst = src if in_place else src.new_empty(src.shape)
            ctx.xts_crypt(kh, dir, src, dst, du, first)
            assert np.array_equal(to_np(dst), ref), (bits, dir, du, units, in_place)
    finally:
        ctx.delkey(kh)


def test_long_units_batched(ctx):
    import paper_1305_3345_gb300 as kg
    du, units = 8193 * 16, 5
    key = w.xts_key(62, 256)
    data = w.seeded_bytes(62, w.STREAM_DATA, du * units)
    kh = ctx.setkey(key, True)
    try:
        src = to_dev(data)
        dst = src.new_empty(src.shape)
        r = np.zeros(1, dtype=kg.request_dtype())
        r["mode"], r["key"], r["len"], r["unit_size"] = w.MODE_XTS, kh, du * units, du
        r["src"], r["dst"], r["sector"] = src.data_ptr(), dst.data_ptr(), 5
        assert ctx.poll(ctx.submit(r)) == 0
        assert np.array_equal(to_np(dst), oracle.xts(key, 0, data, du, 5))
    finally:
        ctx.delkey(kh)


@pytest.mark.parametrize("mib", [64, 256])  # on the tables; with bit-planes
def test_long_units_cost_no_more_time(ctx, mib):
    """A unit of 2^20 blocks against units of 256: a jump of a step per 32 blocks
    made such a call take four to six times as long."""
    import torch
    kh = ctx.setkey(w.xts_key(63, 256), True)
    src = torch.zeros(mib << 20, dtype=torch.uint8, device="cuda")
    dst = torch.zeros_like(src)

    def best(du):
        ms = []
        for _ in range(8):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            for _ in range(4):
                ctx.xts_crypt(kh, 0, src, dst, du, 1)
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms[2:])

    try:
        long, short = best(16 << 20), best(4096)
        assert long < 1.5 * short, (long, short)
    finally:
        ctx.delkey(kh)


def test_long_units_served(ctx):
    import paper_1305_3345_gb300 as kg
    du, units = (1 << 20) + 16, 3
    key = w.xts_key(64, 128)
    data = w.seeded_bytes(64, w.STREAM_DATA, du * units)
    kh = ctx.setkey(key, True)
    src = to_dev(data)
    dst = src.new_empty(src.shape)
    r = np.zeros(1, dtype=kg.request_dtype())
    r["mode"], r["key"], r["len"], r["unit_size"], r["dir"] = w.MODE_XTS, kh, du * units, du, 1
    r["src"], r["dst"], r["sector"] = src.data_ptr(), dst.data_ptr(), 5
    import torch
    torch.cuda.synchronize()
    ctx.serve_start()
    try:
        rc, status, _ = ctx.serve_poll(ctx.serve_submit(r))
        assert rc == 0 and status == 0
    finally:
        ctx.serve_stop()
    assert np.array_equal(to_np(dst), oracle.xts(key, 1, data, du, 5))
    ctx.delkey(kh)
