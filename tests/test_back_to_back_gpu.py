"""Calls queued one behind the other, each reading what the one before wrote:
the bulk kernels start before their predecessor in the stream has finished (for
their table fills) and must not touch a buffer before it has.  Checked eagerly,
captured in a CUDA graph and across streams, against the CPU oracle."""
import numpy as np
import pytest

import oracle
import workloads as w
from conftest import to_dev, to_np

pytestmark = pytest.mark.gpu

# bytes of each call on the front of one buffer, at an offset that is 16-byte
# but not 32-byte aligned: small after large and large after small
STEPS = [("xts", 0, 96 * 4096), ("cbc_enc", 0, 4096), ("cbc_dec", 1, 300 * 4096), ("ecb", 0, 512),
         ("xts", 1, 4096), ("cts", 0, 520 * 640), ("cbc_enc", 0, 640 * 512), ("ecb", 1, 300 * 4096),
         ("cts", 1, 520 * 3), ("cbc_dec", 1, 512), ("xts", 0, 300 * 4096)]
N = 300 * 4096


@pytest.fixture(scope="module")
def setup(ctx):
    xk, ck = w.xts_key(41, 256), w.single_key(41, 128)
    ivs = w.page_ivs(41, N // 512)
    data = w.seeded_bytes(41, w.STREAM_DATA, N)
    x, c = ctx.setkey(xk, True), ctx.setkey(ck, False)
    want = data.copy()
    for kind, dir, n in STEPS:
        part = want[:n]
        unit = 520 if kind == "cts" else 512
        if kind in ("xts", "cts"):
            want[:n] = oracle.xts(xk, dir, part, unit, 7)
        elif kind == "ecb":
            want[:n] = oracle.ecb(ck, dir, part)
        else:
            want[:n] = oracle.cbc(ck, dir, part, 512, ivs[:n // 512])
    yield ctx, x, c, to_dev(np.ascontiguousarray(ivs).reshape(-1)), data, want
    ctx.delkey(x)
    ctx.delkey(c)


def chain(ctx, x, c, iv, buf):
    for kind, dir, n in STEPS:
        b = buf[:n]
        if kind in ("xts", "cts"):
            ctx.xts_crypt(x, dir, b, b, 520 if kind == "cts" else 512, 7)
        elif kind == "ecb":
            ctx.ecb_crypt(c, dir, b, b)
        elif dir == 1:
            ctx.cbc_decrypt(c, b, b, 512, iv[:n // 32])
        else:
            ctx.cbc_encrypt_pages(c, b, b, 512, iv[:n // 32])


def fresh(data):
    import torch
    buf = torch.empty(N + 16, dtype=torch.uint8, device="cuda")[16:]
    buf.copy_(to_dev(data))
    return buf


def test_chain_in_place(setup):
    ctx, x, c, iv, data, want = setup
    for _ in range(10):
        buf = fresh(data)
        chain(ctx, x, c, iv, buf)
        assert np.array_equal(to_np(buf), want)


def test_chain_captured(setup):
    import torch
    ctx, x, c, iv, data, want = setup
    start, buf = fresh(data), fresh(data)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        buf.copy_(start)
        chain(ctx, x, c, iv, buf)
    for _ in range(5):
        buf.zero_()
        g.replay()
        assert np.array_equal(to_np(buf), want)


def test_chain_across_streams(setup):
    """Each call on another stream than the one before, ordered by events."""
    import torch
    ctx, x, c, iv, data, want = setup
    streams = [torch.cuda.Stream() for _ in range(3)]
    buf = fresh(data)
    torch.cuda.synchronize()
    ev = None
    for i, (kind, dir, n) in enumerate(STEPS):
        s = streams[i % 3]
        if ev is not None:
            s.wait_event(ev)
        b = buf[:n]
        if kind in ("xts", "cts"):
            ctx.xts_crypt(x, dir, b, b, 520 if kind == "cts" else 512, 7, stream=s)
        elif kind == "ecb":
            ctx.ecb_crypt(c, dir, b, b, stream=s)
        elif dir == 1:
            ctx.cbc_decrypt(c, b, b, 512, iv[:n // 32], stream=s)
        else:
            ctx.cbc_encrypt_pages(c, b, b, 512, iv[:n // 32], stream=s)
        ev = torch.cuda.Event()
        ev.record(s)
    torch.cuda.synchronize()
    assert np.array_equal(to_np(buf), want)
