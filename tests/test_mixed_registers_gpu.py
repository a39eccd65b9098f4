"""The register count that the mixed kernels' register shares are drawn from:
what they were compiled to, and what a library does whose compiler gave another
one (it must start, and large calls must run on the tables)."""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

LARGE_CALLS = """
import numpy as np, torch
import paper_1305_3345_gb300 as kg, oracle, workloads as w
with kg.Context(0) as c:
    n = 104 << 20
    data = w.seeded_bytes(97, w.STREAM_DATA, n)
    src = torch.from_numpy(data.copy()).cuda()
    dst = torch.zeros_like(src)
    key = w.xts_key(97, 256)
    c.xts_crypt(c.setkey(key, True), 0, src, dst, 4096, 3)
    assert np.array_equal(dst.cpu().numpy(), oracle.xts(key, 0, data, 4096, 3))
    key, ivs = w.single_key(97, 128), w.page_ivs(97, n // 4096)
    c.cbc_decrypt(c.setkey(key, False), src, dst, 4096, torch.from_numpy(ivs.reshape(-1).copy()).cuda())
    assert np.array_equal(dst.cpu().numpy(), oracle.cbc(key, 1, data, 4096, ivs))
print("large calls equal the oracle")
"""


@pytest.fixture(scope="module")
def child(tmp_path_factory):
    cc = shutil.which("gcc")
    if not cc:
        pytest.skip("gcc is not available")
    shim = str(tmp_path_factory.mktemp("shim") / "func_attributes_shim.so")
    subprocess.run([cc, "-shared", "-fPIC", "-O1", "-I/usr/local/cuda/include",
                    os.path.join(HERE, "func_attributes_shim.c"), "-o", shim, "-ldl"], check=True)

    def run(regs):
        env = dict(os.environ, LD_PRELOAD=shim, PYTHONPATH=ROOT)
        if regs:
            env["SHIM_REGS"] = str(regs)
        return subprocess.run([sys.executable, "-c", LARGE_CALLS], cwd=ROOT, env=env, capture_output=True, text=True,
                              timeout=300)
    return run


def test_compiled_register_count(child):
    r = child(None)
    assert r.returncode == 0 and "equal the oracle" in r.stdout, r.stderr
    seen = [line for line in r.stderr.splitlines() if line.startswith("shim:")]
    assert len(seen) >= 13 and set(seen) == {"shim: 96 registers"}, seen


def test_another_register_count_stays_on_the_tables(child):
    r = child(104)
    assert r.returncode == 0 and "equal the oracle" in r.stdout, r.stderr
