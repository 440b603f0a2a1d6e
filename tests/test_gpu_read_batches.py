"""Batches of cached reads (gfs_read_many) against reading the same requests one by one.

A latency trace turns batches off, so the same calls on a context with one take the general
path.  One block serves the requests in order: the delivered bytes, the return values, the
counters and the request and eviction traces then have one right value, and both paths must
reach it, through a cache that recycles its frames as well as one that does not.
"""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
KiB = 1024


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    torch.cuda.init()
    return torch


@pytest.fixture(scope="module")
def gfs():
    from paper_2109_05366_gb300 import gfs as g
    g.load()
    return g


def _requests(size, page, seed):
    """(offset, length, destination) with repeated and neighbouring pages, page ends, empty
    reads, reads cut by and past the end of the file, reads of more pages than a batch
    holds, and destinations that meet an earlier read's."""
    rng = np.random.default_rng(seed)
    got, pos = [], 0
    for i in range(400):
        kind = i % 20
        n = int(rng.integers(1, 3 * page // 2))
        o = int(rng.integers(0, size))
        if kind == 3:
            n = 0
        elif kind == 5:
            o = size + int(rng.integers(0, 99))
        elif kind == 7:
            o = size - 5
        elif kind == 9:
            o, n = o // page * page, page
        elif kind in (10, 11, 12, 13):
            o, n = 2 * page - 40 + 7 * kind, 64
        elif kind == 15:
            o, n = min(o, size // 2), 34 * page + 3
        d = pos + int(rng.integers(0, 16))
        if kind in (12, 17) and got:
            d = max(0, got[-1][2] - 9)
        got.append((o, n, d))
        pos = max(pos, d + n)
    return got, pos + 16


@pytest.mark.parametrize("page,frames,threads,advice", [
    (4 * KiB, 256, 128, 2), (4 * KiB, 64, 128, 2), (4 * KiB, 64, 256, 0), (64 * KiB, 64, 128, 2), (64 * KiB, 40, 512, 0),
])
def test_batches_equal_single_reads(torch_cuda, gfs, datadir, page, frames, threads, advice):
    torch = torch_cuda
    size = 48 * page + 1237
    ref = np.random.default_rng(11).integers(0, 256, size, dtype=np.uint8)
    path = os.path.join(datadir, "batches_%d.bin" % page)
    ref.tofile(path)
    reqs, room = _requests(size, page, 12)
    want = np.full(room, 0xA5, dtype=np.uint8)
    for o, n, d in reqs:
        part = ref[o:o + n]
        want[d:d + len(part)] = part
    off, ln, dst = (torch.tensor([r[k] for r in reqs], dtype=torch.int64, device="cuda") for k in range(3))
    seen = []
    for lat in (0, 1 << 14):
        with gfs.Context(cache_bytes=frames * page, page_size=page, latency_capacity=lat, trace_capacity=1 << 14) as ctx:
            fid = ctx.open(path)
            ctx.fadvise(fid, advice)
            for _ in range(2):
                buf = torch.full((room,), 0xA5, dtype=torch.uint8, device="cuda")
                ret = torch.full((len(reqs),), -999, dtype=torch.int64, device="cuda")
                ctx.read_many(fid, off, ln, dst, buf, ret, blocks=1, threads=threads)
                torch.cuda.synchronize()
                assert ret.cpu().tolist() == [max(0, min(n, size - o)) for o, n, _ in reqs]
                assert np.array_equal(buf.cpu().numpy(), want)
            st = ctx.stats()
            seen.append(([st[k] for k in ("greads", "hits", "misses", "rpcs", "pages_fetched", "evictions",
                                          "unconsumed_evictions", "ra_pages_sync", "ra_pages_async", "timeouts")],
                         ctx.trace()))
    assert seen[0] == seen[1]


@pytest.mark.parametrize("frames", [8, 64])
def test_batches_of_many_blocks_share_pages(torch_cuda, gfs, datadir, frames):
    """Blocks pin the same few pages in batches while others read pages in and evict them."""
    torch = torch_cuda
    page, size = 4 * KiB, 24 * 4 * KiB + 7
    ref = np.random.default_rng(13).integers(0, 256, size, dtype=np.uint8)
    path = os.path.join(datadir, "batches_shared.bin")
    ref.tofile(path)
    rng = np.random.default_rng(14)
    n = 6000
    o = rng.integers(0, size, n)
    ln = rng.integers(0, 900, n)
    d = np.arange(n) * 1024 + rng.integers(0, 16, n)
    t = lambda a: torch.from_numpy(a.astype(np.int64)).cuda()  # noqa: E731
    with gfs.Context(cache_bytes=frames * page, page_size=page) as ctx:
        fid = ctx.open(path)
        ctx.fadvise(fid, gfs.ADV_RANDOM)
        buf = torch.zeros(n * 1024 + 1024, dtype=torch.uint8, device="cuda")
        ret = torch.zeros(n, dtype=torch.int64, device="cuda")
        ctx.read_many(fid, t(o), t(ln), t(d), buf, ret, blocks=40, threads=128)
        torch.cuda.synchronize()
        st = ctx.stats()
    buf, ret = buf.cpu().numpy(), ret.cpu().numpy()
    for i in range(n):
        part = ref[o[i]:o[i] + ln[i]]
        assert ret[i] == len(part)
        assert np.array_equal(buf[d[i]:d[i] + len(part)], part)
    assert st["greads"] == n and st["timeouts"] == 0


@pytest.mark.parametrize("lat", [0, 16])
def test_a_cached_page_read_over_and_over_is_queued_once(torch_cuda, gfs, datadir, lat):
    """4 GiB of reads of a page and more must not count it as newly consumed again."""
    torch = torch_cuda
    page, n, passes = 4 * KiB, 1 << 17, 80  # 2^32 bytes are eight passes
    path = os.path.join(datadir, "batches_wrap.bin")
    np.random.default_rng(15).integers(0, 256, page, dtype=np.uint8).tofile(path)
    with gfs.Context(cache_bytes=4 * page, page_size=page, latency_capacity=lat, timeout_ns=200_000_000) as ctx:
        fid = ctx.open(path)
        ctx.fadvise(fid, gfs.ADV_RANDOM)
        off = torch.zeros(n, dtype=torch.int64, device="cuda")
        buf = torch.zeros(n * page, dtype=torch.uint8, device="cuda")
        ret = torch.zeros(n, dtype=torch.int64, device="cuda")
        dst = torch.arange(n, dtype=torch.int64, device="cuda") * page
        for _ in range(passes):
            ctx.read_many(fid, off, torch.full_like(off, page), dst, buf, ret, blocks=608, threads=128)
        torch.cuda.synchronize()
        st = ctx.stats()
    assert st["timeouts"] == 0  # (blocks that race for the page at first may evict it once: not what this is about)
    assert st["hits"] + st["misses"] >= n * passes and (ret == page).all()
