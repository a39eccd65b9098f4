"""One request on registered host pages, which cross the host link: bit-exact
against the CPU oracle in every form, and as fast as the link's whole lines."""
import time

import numpy as np
import pytest

import oracle
import workloads as w
from test_dispatch_gpu import HostPages, request

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,unit,pages", [
    (128, 4096, 32), (128, 4096, 33), (192, 512, 128), (192, 512, 129), (256, 128, 256), (256, 128, 257),
    (128, 4096, 1100), (256, 640, 5000), (256, 4112, 300), (192, 48, 2000),
])
def test_cbc_encryption_over_the_link(ctx, bits, unit, pages):
    import paper_1305_3345_gb300 as kg
    key = w.single_key(91, bits)
    kh = ctx.setkey(key, False)
    hp = HostPages(ctx, 91 + unit, unit * pages, unit)
    try:
        ref = oracle.cbc(key, 0, hp.data, unit, hp.ivs_np[:pages])
        for out in (hp.dst, hp.src):  # out of place, then in place
            r = request(kg, kg.MODE_CBC_ENC, kh, hp.src.data_ptr(), out.data_ptr(), unit * pages, unit,
                        ivs=hp.ivs.data_ptr())
            assert ctx.crypt(r, kg.DISPATCH_GPU) == (0, kg.DISPATCH_GPU)
            assert np.array_equal(out.numpy(), ref), (bits, unit, pages)
    finally:
        hp.close()
        ctx.delkey(kh)


def test_cbc_encryption_over_the_link_is_link_bound(ctx):
    """64 MiB at 65 GB/s or more; 16 bytes a page at a time reach 34."""
    import paper_1305_3345_gb300 as kg
    size = 64 << 20
    kh = ctx.setkey(w.single_key(92, 128), False)
    hp = HostPages(ctx, 92, size)
    try:
        r = request(kg, kg.MODE_CBC_ENC, kh, hp.src.data_ptr(), hp.dst.data_ptr(), size, 4096, ivs=hp.ivs.data_ptr())
        times = []
        for _ in range(8):
            t = time.perf_counter()
            assert ctx.crypt(r, kg.DISPATCH_GPU)[0] == 0
            times.append(time.perf_counter() - t)
        assert size / min(times) > 65e9, size / min(times)
    finally:
        hp.close()
        ctx.delkey(kh)


@pytest.mark.parametrize("bits,dir,du,mib", [(128, 1, 512, 48), (256, 0, 4096, 96), (256, 1, 528, 48)])
def test_host_call_at_the_line_between_sm_counts(ctx, bits, dir, du, mib):
    """Registered pages just up to and past the size from which more SMs run."""
    import torch
    key = w.xts_key(93, bits)
    kh = ctx.setkey(key, True)
    units = (mib << 20) // du + 1
    data = w.seeded_bytes(93 + du, w.STREAM_DATA, du * units)
    src = torch.from_numpy(data.copy()).pin_memory()
    dst = torch.zeros(du * units, dtype=torch.uint8).pin_memory()
    ref = oracle.xts(key, dir, data, du, 9)
    ctx.host_register(src)
    ctx.host_register(dst)
    try:
        for n in (units - 1, units):
            dst.zero_()
            ctx.xts_crypt_host(kh, dir, src[:n * du], dst[:n * du], du, 9)
            assert np.array_equal(dst.numpy()[:n * du], ref[:n * du]), (bits, dir, du, n)
    finally:
        ctx.host_unregister(src)
        ctx.host_unregister(dst)
        ctx.delkey(kh)


@pytest.mark.parametrize("bits,unit,pages", [(128, 4096, 511), (256, 4096, 513), (192, 528, 9000), (128, 512, 98305)])
def test_cbc_decryption_over_the_link(ctx, bits, unit, pages):
    import paper_1305_3345_gb300 as kg
    key = w.single_key(94, bits)
    kh = ctx.setkey(key, False)
    hp = HostPages(ctx, 94 + unit, unit * pages, unit)
    try:
        ref = oracle.cbc(key, 1, hp.data, unit, hp.ivs_np[:pages])
        for out in (hp.dst, hp.src):  # out of place, then in place
            r = request(kg, kg.MODE_CBC_DEC, kh, hp.src.data_ptr(), out.data_ptr(), unit * pages, unit,
                        ivs=hp.ivs.data_ptr())
            assert ctx.crypt(r, kg.DISPATCH_GPU) == (0, kg.DISPATCH_GPU)
            assert np.array_equal(out.numpy(), ref), (bits, unit, pages)
    finally:
        hp.close()
        ctx.delkey(kh)
