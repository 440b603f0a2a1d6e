"""The workloads whose speed this repository answers for.

Each case is one call (or the few calls that belong together) of the public Python
binding, on files that a case makes itself under /dev/shm: bytes uniform on 0..255,
float32 uniform on [-1, 1), int32 from a Zipf law (s = 1.1) -- the distributions of the
benchmark's workloads.  Files are unlinked as soon as they are open.

  scan       the stride scan (count, byte sum, position hash per stride).  Not resident:
             the cache is cleared first, so every byte crosses the host link, and a cache
             smaller than the file recycles its frames on the way.  Resident: the file is
             in the GPU page cache from an earlier pass, as in every epoch after the first.
  reads      independent greads into one buffer (gather of tiles or of records).
  rowdot     row-major float32 matrix times a resident vector.
  histogram  counts of an int32 file.
  serve      the serving loop: start, submit scans of files of uneven size, collect every
             completion, stop.
"""
from __future__ import annotations

import math
import os
import tempfile
import threading

import numpy as np
import torch

from paper_2109_05366_gb300 import gfs

KiB, MiB, GiB = 1 << 10, 1 << 20, 1 << 30
NBINS = 1 << 20


def listed():
    scan = dict(kind="scan", resident=False, host=False, xfer=gfs.XFER_MAPPED, mode=gfs.MODE_READAHEAD, fused=False,
                threads=256)
    reads = dict(kind="reads", mode=gfs.MODE_READAHEAD, threads=128, blocks=1216)
    return [
        # the smallest call: a file of about a megabyte that is already on the GPU, strides
        # that are no power of two, results wanted on the host
        dict(scan, name="small_file_again", resident=True, host=True, fused=True, size=1234567, page=64 * KiB,
             cache=4 * MiB, stride=96 * KiB + 8, blocks=16),
        # the first pass over a file that fits the cache (the 64 MiB workload of the benchmark)
        dict(scan, name="first_pass_64m", size=64 * MiB, page=256 * KiB, cache=128 * MiB, stride=MiB, blocks=64),
        # one pass over a file larger than the cache, large pages: the benchmark's shape
        dict(scan, name="stream_1g", size=GiB, page=512 * KiB, cache=384 * MiB, stride=MiB, blocks=296),
        # the same with the paper's page size
        dict(scan, name="stream_4k_pages", size=GiB, page=4 * KiB, cache=256 * MiB, stride=MiB, blocks=296),
        # a file that the GPU cannot map (cold or direct files): host threads pread, the GPU copies
        dict(scan, name="stream_staged", size=256 * MiB, page=256 * KiB, cache=160 * MiB, stride=MiB, blocks=64,
             xfer=gfs.XFER_PULL),
        # later epochs over a data set that stays on the GPU, default consumer
        dict(scan, name="epoch_1g", resident=True, size=GiB, page=512 * KiB, cache=GiB + 256 * MiB, stride=MiB,
             blocks=296),
        # later epochs with small pages (one cache that also serves small random reads)
        dict(scan, name="epoch_4k_pages", resident=True, fused=True, size=256 * MiB + 777, page=4 * KiB,
             cache=384 * MiB, stride=MiB, blocks=296),
        # random tiles of a database, one page each, nothing cached yet
        dict(reads, name="tiles_4k", resident=False, size=GiB, page=4 * KiB, cache=GiB, n=1 << 17, lo=4 * KiB,
             hi=4 * KiB, align=4 * KiB),
        # records of uneven length at any byte of a file that is cached (batches of training samples)
        dict(reads, name="records_cached", resident=True, size=512 * MiB, page=64 * KiB, cache=640 * MiB, n=16384,
             lo=256, hi=64 * KiB, align=1),
        # matrix times vector again and again (an iterative solver): the matrix stays cached
        dict(kind="rowdot", name="rowdot_again", resident=True, rows=16384, cols=8192, stripe=64, page=512 * KiB,
             cache=640 * MiB, blocks=296),
        # one pass of counting over a file
        dict(kind="histogram", name="histogram_256m", resident=False, size=256 * MiB, page=512 * KiB,
             cache=512 * MiB, blocks=296),
        # serving: scans of files of uneven size that arrive together and share one cache
        dict(kind="serve", name="serve_mix", files=6, requests=24, lo=MiB, hi=64 * MiB, page=512 * KiB, cache=GiB,
             ctas=296, unit=MiB),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _up(n, m):
    return (n + m - 1) // m * m


def draw(rng):
    kind = rng.choice(["first", "first", "staged", "again", "again", "again", "reads", "reads", "reads", "rowdot",
                       "histogram", "serve"])
    if kind in ("first", "staged", "again"):
        blocks = rng.choice([16, 64, 148, 296, 592])
        page = rng.choice([64, 256, 512] if kind == "staged" else [4, 16, 64, 256, 512, 1024]) * KiB
        mode = rng.choice([gfs.MODE_READAHEAD] * 3 + [gfs.MODE_ONDEMAND])
        stride = _log(rng, 16 * KiB, 2 * MiB)
        odd = rng.random() < 1 / 3
        stride = stride | 1 if odd else _up(stride, 4 * KiB)
        top = min(GiB, blocks * 2 * MiB)
        if odd or kind == "staged" or mode == gfs.MODE_ONDEMAND or page < 16 * KiB:
            top = min(top, 128 * MiB)
        size = _log(rng, 256 * KiB, top)
        held = blocks * (_up(stride, page) + page)  # pages that the running greads touch at once
        fits = kind == "again" or rng.random() < 0.5
        cache = _up(size + size // 4, page) + 16 * page if fits else max(_up(size // 4, page), 2 * held)
        return dict(kind="scan", resident=kind == "again", host=rng.random() < 0.25, fused=rng.random() < 0.5,
                    xfer=gfs.XFER_PULL if kind == "staged" else gfs.XFER_MAPPED, mode=mode, size=size, page=page,
                    cache=cache, stride=stride, blocks=blocks, threads=rng.choice([128, 256, 256, 512]))
    if kind == "reads":
        page = rng.choice([4, 4, 16, 64, 256]) * KiB
        resident = rng.random() < 0.6
        lo = _log(rng, 64, 16 * KiB)
        hi = min(lo * rng.choice([1, 4, 64]), 128 * KiB)
        size = _log(rng, 4 * MiB, 512 * MiB)
        per_read = (lo + hi) // 2 + (0 if resident else 2 * page)
        n = min(_log(rng, 64, 1 << 17), max(64, 256 * MiB // per_read))
        blocks, threads = rng.choice([(1216, 128), (1216, 128), (592, 256), (296, 256)])
        align = rng.choice([1, 4, 4096])
        return dict(kind="reads", resident=resident, mode=rng.choice([gfs.MODE_READAHEAD, gfs.MODE_ONDEMAND]),
                    size=size, page=page, cache=_up(size + size // 4, page) + 16 * page, n=n, lo=lo, hi=hi,
                    align=align, blocks=blocks, threads=threads)
    resident = rng.random() < 0.5
    page = rng.choice([64, 256, 512]) * KiB
    if kind == "rowdot":
        cols = 4 * _log(rng, 256, 8192)
        rows = max(64, _log(rng, 4 * MiB, 256 * MiB) // (4 * cols))
        return dict(kind="rowdot", resident=resident, rows=rows, cols=cols, stripe=rng.choice([32, 64, 128]),
                    page=page, cache=_up(5 * rows * cols, page) + 16 * page, blocks=296)
    if kind == "histogram":
        size = 4 * _log(rng, MiB, 64 * MiB)
        return dict(kind="histogram", resident=resident, size=size, page=page, cache=_up(size + size // 4, page) + 16 * page,
                    blocks=296)
    return dict(kind="serve", files=rng.randint(2, 8), requests=rng.randint(4, 32), lo=512 * KiB,
                hi=_log(rng, 4 * MiB, 48 * MiB), page=page, cache=GiB, ctas=rng.choice([152, 296]),
                unit=rng.choice([256 * KiB, MiB]))


# ---------------------------------------------------------------- inputs
def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 16 + salt)
    return g


def _bytes(n, seed, salt=0):
    """n uniform bytes (device)."""
    words = torch.randint(-(1 << 63), (1 << 63) - 1, ((n + 7) // 8,), generator=_gen(seed, salt), device="cuda")
    return words.view(torch.uint8)[:n]


def _matrix(case, seed):
    return torch.rand(case["rows"], case["cols"], generator=_gen(seed), device="cuda") * 2 - 1


def _vector(case, seed):
    return torch.rand(case["cols"], generator=_gen(seed, 1), device="cuda") * 2 - 1


def _zipf(n, seed):
    cdf = torch.arange(1, NBINS + 1, dtype=torch.float64, device="cuda").pow(-1.1).cumsum(0)
    cdf /= cdf[-1].clone()
    u = torch.rand(n, generator=_gen(seed), dtype=torch.float64, device="cuda")
    return torch.searchsorted(cdf, u, right=True).clamp_(max=NBINS - 1).to(torch.int32)


def _lengths(case, seed):
    """Log-uniform lengths between lo and hi, every seed in an order of its own."""
    n = case["n"]
    u = (torch.randperm(n, generator=_gen(seed, 2), device="cuda").to(torch.float64) + 0.5) / n
    return (case["lo"] * (case["hi"] / case["lo"]) ** u).to(torch.int64)


def _reads(case, seed):
    """(offsets, lengths, destinations, buffer bytes); destinations are 16-byte aligned."""
    ln = _lengths(case, seed)
    u = torch.rand(case["n"], generator=_gen(seed, 3), dtype=torch.float64, device="cuda")
    off = ((case["size"] - ln).clamp(min=0).to(torch.float64) * u).to(torch.int64)
    off -= off % case["align"]
    room = (ln + 15) // 16 * 16
    end = room.cumsum(0)
    return off, ln, end - room, int(end[-1])


def _file_sizes(case, seed):
    rng = np.random.default_rng(seed)
    return [int(v) for v in np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["files"]))]


def _requests(case, seed):
    """(file, offset, length) of every serving request: whole files, and some tails."""
    rng, sizes = np.random.default_rng(seed + 1), _file_sizes(case, seed)
    got = []
    for i in range(case["requests"]):
        f = i % case["files"]
        off = int(rng.integers(0, sizes[f] // 2)) if i % 4 == 3 else 0
        got.append((f, off, sizes[f] - off))
    return got


def _write(data):
    """A new file under /dev/shm holding the device tensor's bytes; its path."""
    host = data.reshape(-1).view(torch.uint8).cpu().numpy()
    fd, path = tempfile.mkstemp(prefix="gfs_case_", dir="/dev/shm")
    step = max(MiB, -(-host.size // 16))

    def part(a):
        b = min(a + step, host.size)
        while a < b:
            a += os.pwrite(fd, host[a:b], a)

    try:
        ts = [threading.Thread(target=part, args=(a,)) for a in range(0, host.size, step)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
    finally:
        os.close(fd)
    return path


class State:
    def __init__(self, case, **cfg):
        self.case = case
        self.ctx = gfs.Context(cache_bytes=case["cache"] // case["page"] * case["page"], page_size=case["page"],
                               rpc_slots=512, **cfg)
        self.fids = []

    def add(self, data):
        path = _write(data)
        try:
            self.fids.append(self.ctx.open(path))
        finally:
            os.unlink(path)
        return self.fids[-1]


def prepare(case, seed):
    kind, page = case["kind"], case["page"]
    # request and readahead sizes as the benchmark configures them: 16 pages of the large sizes, 64 of the small
    cfg = dict(max_rpc_pages=min(64, max(16, MiB // page)), ra_cap_pages=min(63, max(8, 256 * KiB // page - 1)))
    s = State(case, mode=case.get("mode", gfs.MODE_READAHEAD), xfer=case.get("xfer", gfs.XFER_MAPPED), **cfg)
    if kind == "serve":
        for i, n in enumerate(_file_sizes(case, seed)):
            s.add(_bytes(n, seed, i))
        s.requests = _requests(case, seed)
        return s
    if kind == "rowdot":
        s.add(_matrix(case, seed))
        s.vec = _vector(case, seed)
    elif kind == "histogram":
        s.add(_zipf(case["size"] // 4, seed))
    else:
        s.add(_bytes(case["size"], seed))
    if kind == "scan":
        ns = -(-case["size"] // case["stride"])
        s.out = None if case["host"] else tuple(torch.empty(ns, dtype=torch.int64, device="cuda") for _ in range(3))
    if kind == "reads":
        s.ctx.fadvise(s.fids[0], gfs.ADV_RANDOM)
        s.off, s.len, s.dst, n = _reads(case, seed)
        s.buf = torch.zeros(n, dtype=torch.uint8, device="cuda")
        s.ret = torch.zeros(case["n"], dtype=torch.int64, device="cuda")
    if case.get("resident"):  # an earlier pass over the file has brought it into the cache
        s.ctx.scan(s.fids[0], max(page, 256 * KiB), blocks=64, fused=True)
        torch.cuda.synchronize()
    return s


def run(s):
    case, ctx = s.case, s.ctx
    kind = case["kind"]
    if kind == "serve":
        return _serve(s)
    if not case["resident"]:
        ctx.reset_cache()
    fid = s.fids[0]
    if kind == "scan":
        args = dict(stride=case["stride"], blocks=case["blocks"], threads=case["threads"], fused=case["fused"])
        if case["host"]:
            return [a.view(np.int64) for a in ctx.scan_host(fid, **args)]
        return ctx.scan(fid, out=s.out, **args)
    if kind == "reads":
        ctx.read_many(fid, s.off, s.len, s.dst, s.buf, s.ret, blocks=case["blocks"], threads=case["threads"])
        return s.buf, s.ret
    if kind == "rowdot":
        row = 4 * case["cols"]
        return ctx.rowdot(fid, case["rows"], case["cols"], s.vec, stripe_rows=case["stripe"],
                          read_len=max(1, MiB // row) * row, blocks=case["blocks"])
    return ctx.histogram(fid, nbins=NBINS, blocks=case["blocks"])


def _serve(s):
    case, ctx = s.case, s.ctx
    ctx.serve_start(ctas=case["ctas"], threads=256, unit_bytes=case["unit"], max_requests=64, queue_slots=64)
    n, done = len(s.requests), {}
    for tag, (f, off, length) in enumerate(s.requests):
        while not ctx.submit_scan(s.fids[f], off, length, tag):
            pass
    while len(done) < n:
        for c in ctx.poll():
            done[c["tag"]] = c
    ctx.serve_stop()
    return [np.array([done[t][k] for t in range(n)], dtype=np.uint64).view(np.int64)
            for k in ("status", "bytes", "sum", "hash")]


# ---------------------------------------------------------------- what a pass has to do
def work(case):
    kind = case["kind"]
    if kind == "scan":
        return {"bytes": case["size"] + 24 * -(-case["size"] // case["stride"]), "flops": 0}
    if kind == "reads":
        lo, hi = case["lo"], case["hi"]
        mean = lo if lo == hi else (hi - lo) / math.log(hi / lo)
        return {"bytes": case["n"] * (2 * mean + 32), "flops": 0}
    if kind == "rowdot":
        n = case["rows"] * case["cols"]
        return {"bytes": 4 * n + 4 * case["cols"] + 4 * case["rows"], "flops": 2 * n}
    if kind == "histogram":
        return {"bytes": case["size"] + 4 * NBINS, "flops": 0}
    mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
    return {"bytes": case["requests"] * mean, "flops": 0}


# ---------------------------------------------------------------- the results by definition
def _sums(data, first=0):
    """Byte sum and position hash (mod 2^64) of a device byte tensor that starts at file offset `first`."""
    total, hashed = 0, 0
    for a in range(0, data.numel(), 64 * MiB):
        b = data[a:a + 64 * MiB].to(torch.int64)
        pos = torch.arange(first + a + 1, first + a + 1 + b.numel(), dtype=torch.int64, device="cuda")
        total += int(b.sum())
        hashed += int((b * pos).sum())
    return total, hashed


def _stride_sums(data, stride):
    n = data.numel()
    ns = -(-n // stride)
    count = torch.full((ns,), stride, dtype=torch.int64, device="cuda")
    count[-1] = n - (ns - 1) * stride
    total, hashed = torch.empty_like(count), torch.empty_like(count)
    rows = max(1, 64 * MiB // stride)
    for r in range(0, ns, rows):
        k = min(rows, ns - r)
        b = torch.zeros(k * stride, dtype=torch.int64, device="cuda")
        part = data[r * stride:(r + k) * stride]
        b[:part.numel()] = part
        pos = torch.arange(r * stride + 1, (r + k) * stride + 1, dtype=torch.int64, device="cuda")
        total[r:r + k] = b.view(k, stride).sum(1)
        hashed[r:r + k] = (b * pos).view(k, stride).sum(1)
    return count, total, hashed


def exact(case, seed):
    kind = case["kind"]
    if kind == "scan":
        return _stride_sums(_bytes(case["size"], seed), case["stride"])
    if kind == "reads":
        data = _bytes(case["size"], seed)
        off, ln, dst, n = _reads(case, seed)
        buf = torch.zeros(n, dtype=torch.uint8, device="cuda")
        for a in range(0, case["n"], 4096):
            o, k, d = off[a:a + 4096], ln[a:a + 4096], dst[a:a + 4096]
            at = torch.arange(int(k.sum()), device="cuda") - torch.repeat_interleave(k.cumsum(0) - k, k)
            buf[torch.repeat_interleave(d, k) + at] = data[torch.repeat_interleave(o, k) + at]
        return buf, ln
    if kind == "rowdot":
        m, v = _matrix(case, seed), _vector(case, seed).double()
        out = torch.cat([m[r:r + 1024].double() @ v for r in range(0, case["rows"], 1024)])
        _, total, hashed = _stride_sums(m.view(-1).view(torch.uint8), case["stripe"] * case["cols"] * 4)
        return out, total, hashed, torch.zeros(1, dtype=torch.int64)
    if kind == "histogram":
        v = _zipf(case["size"] // 4, seed)
        sums = torch.tensor([_sums(v.view(torch.uint8))[0], 0], dtype=torch.int64)
        return torch.bincount(v, minlength=NBINS).to(torch.int32), sums, torch.zeros(1, dtype=torch.int64)
    files = [_bytes(n, seed, i) for i, n in enumerate(_file_sizes(case, seed))]
    got = [_sums(files[f][off:off + n], off) for f, off, n in _requests(case, seed)]
    u64 = (1 << 64) - 1
    cols = [[0] * len(got), [n for _, _, n in _requests(case, seed)], [t for t, _ in got], [h & u64 for _, h in got]]
    return [np.array(c, dtype=np.uint64).view(np.int64) for c in cols]
