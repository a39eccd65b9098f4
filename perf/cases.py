"""Workloads of the page-crypto service, as a program that uses it runs them.

Each case is one call (or one submission and its wait) through the package's
public binding on data the program already holds: the per-call transforms on
device buffers from one page to 1 GiB, the host-buffer call on pinned pages,
a batch of uneven requests, and a burst through the serving ring.  listed()
gives fixed points, draw() further ones over the same ranges.
"""
import math
import random
import weakref

import numpy as np
import torch

import paper_1305_3345_gb300 as kg

KIB, MIB, GIB = 1 << 10, 1 << 20, 1 << 30

_contexts = {}


def _context(name):
    """One context per process and role, as a storage service keeps: "calls"
    for everything that launches on a stream, "ring" for the serving kernel,
    which leaves the GPU again after half a millisecond without requests."""
    if name not in _contexts:
        ctx = kg.Context(0)
        if name == "ring":
            ctx.serve_start(idle_timeout_ns=500_000)
        _contexts[name] = ctx
    return _contexts[name]


class State:
    """What a caller holds between calls: its context, keys, buffers, requests."""

    def __init__(self, case, ctx):
        self.case, self.ctx = case, ctx
        self.keys = []
        # the keys of a state that is dropped leave the context's key table
        weakref.finalize(self, _drop_keys, ctx, self.keys).atexit = False

    def key(self, raw, xts):
        k = self.ctx.setkey(raw, xts)
        self.keys.append(k)
        return k


def _drop_keys(ctx, keys):
    for k in keys:
        ctx.delkey(k)


def listed():
    return [
        # one page written by a file system: the smallest call
        {"name": "xts256_enc_4k", "kind": "xts", "bits": 256, "dir": 0, "unit": 4096, "units": 1},
        # the service's basic workload: 256 sectors read back, 1 MiB
        {"name": "xts256_dec_1m", "kind": "xts", "bits": 256, "dir": 1, "unit": 4096, "units": 256},
        # bulk encryption of 262,144 sectors, 1 GiB: the headline workload and the largest
        {"name": "xts256_enc_1g", "kind": "xts", "bits": 256, "dir": 0, "unit": 4096, "units": 262144},
        # a read of 512-byte disk sectors, 32 MiB and one sector
        {"name": "xts128_dec_512b", "kind": "xts", "bits": 128, "dir": 1, "unit": 512, "units": 65537},
        # sectors with protection data (520 bytes): units ending in ciphertext stealing, 16 MiB
        {"name": "xts256_enc_520b", "kind": "xts", "bits": 256, "dir": 0, "unit": 520, "units": 32768},
        # file pages read back, 64 MiB and a few pages
        {"name": "cbc128_dec_64m", "kind": "cbc_dec", "bits": 128, "unit": 4096, "units": 16387},
        # a small write of file pages: 256 chains, 1 MiB
        {"name": "cbc256_enc_1m", "kind": "cbc_enc", "bits": 256, "unit": 4096, "units": 256},
        # bulk page encryption, 262,144 chains, 1 GiB
        {"name": "cbc128_enc_1g", "kind": "cbc_enc", "bits": 128, "unit": 4096, "units": 262144},
        # the paper's own mode at a middling size of its sweep
        {"name": "ecb128_enc_256k", "kind": "ecb", "bits": 128, "dir": 0, "unit": 16, "units": 16384},
        # 1,000 uneven requests of many keys and mixed modes in one submission
        {"name": "batch_1000", "kind": "batch", "requests": 1000, "lo": 4 * KIB, "hi": 8 * MIB, "keys": 256},
        # pinned host pages through the copy pipeline, 64 MiB
        {"name": "host_xts256_64m", "kind": "host", "bits": 256, "dir": 0, "unit": 4096, "units": 16384},
        # a burst of 256 requests onto the serving ring
        {"name": "serve_256", "kind": "serve", "requests": 256, "lo": 4 * KIB, "hi": MIB, "keys": 64},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["xts", "cts", "cbc_dec", "cbc_enc", "ecb", "batch", "host", "serve"],
                       [4, 2, 2, 3, 1, 1, 1, 1])[0]
    bits = rng.choice([128, 256])
    if kind == "xts":
        unit = rng.choice([512, 528, 1024, 2048, 4096, 4096, 4112, 8192, 65536])
        return {"kind": "xts", "bits": bits, "dir": rng.randrange(2), "unit": unit,
                "units": max(1, _log(rng, 4 * KIB, 256 * MIB) // unit)}
    if kind == "cts":  # units that are no multiple of 16 bytes, at any byte alignment
        unit = rng.choice([100, 520, 527, 2056, 4097, 4100, 4104])
        return {"kind": "xts", "bits": bits, "dir": rng.randrange(2), "unit": unit,
                "units": max(1, _log(rng, 4 * KIB, 16 * MIB) // unit)}
    if kind in ("cbc_dec", "cbc_enc"):
        bits = rng.choice([128, 192, 256])
        unit = rng.choice([512, 1024, 4096, 4096, 4112, 8192])
        return {"kind": kind, "bits": bits, "unit": unit, "units": max(1, _log(rng, 4 * KIB, 256 * MIB) // unit)}
    if kind == "ecb":
        return {"kind": "ecb", "bits": rng.choice([128, 192, 256]), "dir": rng.randrange(2), "unit": 16,
                "units": _log(rng, 4 * KIB, 256 * MIB) // 16}
    if kind == "host":
        unit = rng.choice([512, 4096])
        return {"kind": "host", "bits": bits, "dir": rng.randrange(2), "unit": unit,
                "units": _log(rng, MIB, 64 * MIB) // unit}
    if kind == "batch":
        return {"kind": "batch", "requests": _log(rng, 16, 1000), "lo": 4 * KIB, "hi": rng.choice([MIB, 8 * MIB]),
                "keys": _log(rng, 4, 256)}
    return {"kind": "serve", "requests": _log(rng, 16, 512), "lo": 4 * KIB, "hi": MIB, "keys": _log(rng, 4, 64)}


def _sizes(case):
    """Request sizes, log-uniform in whole pages: their quantiles, so that
    every seed has the same bytes and only their order differs."""
    q = (np.arange(case["requests"]) + 0.5) / case["requests"]
    s = np.exp(np.log(case["lo"]) + q * (np.log(case["hi"]) - np.log(case["lo"])))
    return 4096 * np.maximum(1, np.rint(s / 4096)).astype(np.int64)


def _total(case):
    return int(_sizes(case).sum()) if "requests" in case else case["unit"] * case["units"]


def work(case):
    """Every payload byte is read once and written once, and every CBC page's
    IV read once; the work itself is table lookups, no floating point."""
    n = _total(case)
    ivs = 16 * case["units"] if case["kind"] in ("cbc_dec", "cbc_enc") else 0
    return {"bytes": 2 * n + ivs, "flops": 0}


def _bytes(gen, n):
    """n uniform random bytes on the GPU."""
    words = torch.randint(-(1 << 63), (1 << 63) - 1, ((n + 7) // 8,), dtype=torch.int64, device="cuda", generator=gen)
    return words.view(torch.uint8)[:n]


def prepare(case, seed):
    kind = case["kind"]
    rng = random.Random("%s %d" % (sorted(case.items()), seed))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rng.getrandbits(62))
    n = _total(case)
    s = State(case, _context("ring" if kind == "serve" else "calls"))
    if kind == "host":
        s.src = torch.empty(n, dtype=torch.uint8, pin_memory=True)
        s.src.copy_(_bytes(gen, n))
        s.dst = torch.zeros(n, dtype=torch.uint8, pin_memory=True)
    else:
        s.src = _bytes(gen, n)
        s.dst = torch.zeros_like(s.src)
    s.sector = rng.getrandbits(40)
    if kind in ("batch", "serve"):
        s.ivs = _bytes(gen, n // 4096 * 16)
        s.reqs = _requests(case, s, rng)
        torch.cuda.synchronize()  # the ring reads what is here now, whatever stream wrote it
    else:
        if kind in ("cbc_dec", "cbc_enc"):
            s.ivs = _bytes(gen, case["units"] * 16)
        xts = kind in ("xts", "host")
        s.k = s.key(rng.randbytes(case["bits"] // 8 * (2 if xts else 1)), xts)
    return s


def _requests(case, s, rng):
    """Half XTS (both directions), a quarter CBC decryption, a quarter CBC
    encryption, spread evenly over the sizes, in random order; AES-128 and
    AES-256 keys, each service key with one for XTS and one for CBC."""
    sizes = _sizes(case)
    r = np.zeros(len(sizes), dtype=kg.request_dtype())
    pattern = np.array([kg.MODE_XTS, kg.MODE_CBC_DEC, kg.MODE_XTS, kg.MODE_CBC_ENC], dtype=np.uint32)
    r["mode"] = pattern[np.arange(len(sizes)) % 4]
    r["dir"] = (np.arange(len(sizes)) // 4) % 2
    r["len"] = sizes
    r["unit_size"] = 4096
    order = list(range(len(sizes)))
    rng.shuffle(order)
    r = r[order]
    off = np.concatenate([[0], np.cumsum(r["len"].astype(np.int64))[:-1]])
    r["src"] = s.src.data_ptr() + off
    r["dst"] = s.dst.data_ptr() + off
    r["ivs"] = np.where(r["mode"] == kg.MODE_XTS, 0, s.ivs.data_ptr() + off // 4096 * 16)
    r["sector"] = [rng.getrandbits(40) for _ in order]
    pairs = []
    for i in range(case["keys"]):
        bits = 128 if i < case["keys"] // 2 else 256
        pairs.append((s.key(rng.randbytes(bits // 4), True), s.key(rng.randbytes(bits // 8), False)))
    which = [pairs[rng.randrange(len(pairs))] for _ in order]
    r["key"] = [p[0] if m == kg.MODE_XTS else p[1] for p, m in zip(which, r["mode"])]
    return r


def run(s):
    c, ctx = s.case, s.ctx
    kind = c["kind"]
    if kind == "xts":
        ctx.xts_crypt(s.k, c["dir"], s.src, s.dst, c["unit"], s.sector)
    elif kind == "ecb":
        ctx.ecb_crypt(s.k, c["dir"], s.src, s.dst)
    elif kind == "cbc_dec":
        ctx.cbc_decrypt(s.k, s.src, s.dst, c["unit"], s.ivs)
    elif kind == "cbc_enc":
        ctx.cbc_encrypt_pages(s.k, s.src, s.dst, c["unit"], s.ivs)
    elif kind == "host":
        ctx.xts_crypt_host(s.k, c["dir"], s.src, s.dst, c["unit"], s.sector)
    elif kind == "batch":
        ctx.poll(ctx.submit(s.reqs))
    else:
        left = s.reqs
        tickets = []
        while len(left):
            _, got = ctx.serve_submit_many(left)
            tickets.extend(got.tolist())
            left = left[len(got):]
        for t in tickets:
            ctx.serve_poll(t)
    return s.dst
