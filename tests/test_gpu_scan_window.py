"""The stride scan's window: reads that end around its edges, reads shorter than it, and the
allocation-free scan of the shortest reads.
"""
import os

import numpy as np
import pytest

from oracle import plain

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


def _bytes_file(datadir, size, seed):
    path = os.path.join(datadir, "sinks_%d_%d.bin" % (size, seed))
    np.random.default_rng(seed).integers(0, 256, size, dtype=np.uint8).tofile(path)
    return path


@pytest.mark.parametrize("threads", [128, 512])
@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("over", [-16, -1, 0, 1, 4096 + 17])
def test_scan_window_edges(torch_cuda, gfs, datadir, threads, fused, over):
    stride = threads // 32 * 16 * KiB + over  # one window of a block of `threads`, and a little
    size = 7 * stride + 4099
    path = _bytes_file(datadir, size, 21)
    want = tuple(list(w) for w in plain.scan_plain(path, stride))
    for page, frames in ((4 * KiB, 4096), (64 * KiB, 24), (512 * KiB, 8)):
        with gfs.Context(cache_bytes=frames * page, page_size=page) as ctx:
            fid = ctx.open(path)
            for _ in range(2):
                got = ctx.scan_host(fid, stride, blocks=3, threads=threads, fused=fused)
                assert tuple(a.tolist() for a in got) == want


@pytest.mark.parametrize("read_len", [1, 15, 17, 255, 256, 4097])
def test_scan_reads_shorter_than_the_window(torch_cuda, gfs, datadir, read_len):
    stride, size = 301, 20011
    path = _bytes_file(datadir, size, 22)
    want = tuple(list(w) for w in plain.scan_plain(path, stride, read_len))
    with gfs.Context(cache_bytes=512 * KiB, page_size=4 * KiB) as ctx:
        fid = ctx.open(path)
        for fused in (False, True):
            got = ctx.scan_host(fid, stride, read_len=read_len, blocks=5, threads=128, fused=fused)
            assert tuple(a.tolist() for a in got) == want


def test_static_scan_of_the_shortest_reads(torch_cuda, gfs, datadir):
    """Reads of 256 bytes at odd offsets in as many blocks as the static array is documented for."""
    import ctypes
    torch = torch_cuda
    stride, blocks = 257, (64 << 20) // 256
    size = 3000 * stride + 5
    path = _bytes_file(datadir, size, 23)
    want = plain.scan_plain(path, stride, 256)
    with gfs.Context(cache_bytes=4 << 20, page_size=4 * KiB, max_streams=4096) as ctx:
        fid = ctx.open(path)
        a = ctx._args(stride, 256, blocks, 128, False, False)
        out = [torch.zeros(len(want[0]), dtype=torch.int64, device="cuda") for _ in range(3)]
        rc = gfs.load().gfs_scan_static(ctx.handle, fid, ctypes.byref(a), *[t.data_ptr() for t in out], None)
        assert rc == 0
        torch.cuda.synchronize()
        for t, w in zip(out, want):
            assert gfs.u64_view(t).tolist() == list(w)
