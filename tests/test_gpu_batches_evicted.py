"""Batches of cached reads while other blocks evict pages: a list goes in batches from the
second launch on a file on, so every case reads once before the lists that are checked.
And reads of many pages into buffers, by many blocks, through a cache smaller than the file."""
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


def _file(datadir, size):
    ref = np.random.default_rng(size).integers(0, 256, size, dtype=np.uint8)
    path = os.path.join(datadir, "evicted_%d.bin" % size)
    ref.tofile(path)
    return path, ref


@pytest.mark.parametrize("advice", [0, 2])
@pytest.mark.parametrize("blocks,threads", [(40, 128), (40, 512), (1216, 128)])
@pytest.mark.parametrize("frames", [8, 64])
def test_batches_under_eviction(torch_cuda, gfs, datadir, frames, blocks, threads, advice):
    torch = torch_cuda
    page, size = 4 * KiB, 24 * 4 * KiB + 7
    path, ref = _file(datadir, size)
    rng = np.random.default_rng(51)
    n = 12000
    t = lambda a: torch.from_numpy(a.astype(np.int64)).cuda()  # noqa: E731
    with gfs.Context(cache_bytes=frames * page, page_size=page) as ctx:
        fid = ctx.open(path)
        ctx.fadvise(fid, advice)
        ctx.scan(fid, 8 * page, blocks=2, threads=128)  # the file has been read: lists go in batches
        torch.cuda.synchronize()
        for _ in range(2):
            o = rng.integers(0, size, n)
            ln = rng.integers(0, 900, n)
            d = np.arange(n) * 1024 + rng.integers(0, 16, n)
            buf = torch.full((n * 1024 + 16,), 0xA5, dtype=torch.uint8, device="cuda")
            ret = torch.full((n,), -999, dtype=torch.int64, device="cuda")
            ctx.read_many(fid, t(o), t(ln), t(d), buf, ret, blocks=blocks, threads=threads)
            torch.cuda.synchronize()
            got = np.minimum(ln, size - o)
            assert np.array_equal(ret.cpu().numpy(), got)
            want = np.full(n * 1024 + 16, 0xA5, dtype=np.uint8)
            for a, k, to in zip(o, got, d):
                want[to:to + k] = ref[a:a + k]
            assert np.array_equal(buf.cpu().numpy(), want)
        st = ctx.stats()
        assert st["timeouts"] == 0
        if frames == 8:  # a third of the file's pages
            assert st["evictions"] > 0


@pytest.mark.parametrize("page", [4 * KiB, 64 * KiB, 512 * KiB])
@pytest.mark.parametrize("threads", [128, 256])
def test_long_reads_through_a_small_cache(torch_cuda, gfs, datadir, page, threads):
    torch = torch_cuda
    size, each, blocks = (24 << 20) + 321, (3 << 20) + 77, 6
    path, ref = _file(datadir, size)
    rng = np.random.default_rng(52)
    n = 14
    off = np.concatenate([[0, size - each, size - 5], rng.integers(0, size - each, n - 3)])
    dst = np.arange(n) * (each + 40) + rng.integers(0, 16, n)
    t = lambda a: torch.from_numpy(a.astype(np.int64)).cuda()  # noqa: E731
    room = blocks * (each // page + 2)  # pages that the running reads touch at once
    with gfs.Context(cache_bytes=min(room, size // 2 // page) * page, page_size=page, max_rpc_pages=16) as ctx:
        fid = ctx.open(path)
        for again in range(2):
            buf = torch.full((n * (each + 40) + 16,), 0xA5, dtype=torch.uint8, device="cuda")
            ret = torch.full((n,), -999, dtype=torch.int64, device="cuda")
            ctx.read_many(fid, t(off), t(np.full(n, each)), t(dst), buf, ret, blocks=blocks, threads=threads)
            torch.cuda.synchronize()
            got = np.minimum(each, size - off)
            assert np.array_equal(ret.cpu().numpy(), got)
            want = np.full(n * (each + 40) + 16, 0xA5, dtype=np.uint8)
            for a, k, to in zip(off, got, dst):
                want[to:to + k] = ref[a:a + k]
            assert np.array_equal(buf.cpu().numpy(), want)
        st = ctx.stats()
        assert st["timeouts"] == 0 and st["evictions"] > 0
