"""Pages handed to their consumer as they arrive from the host: pages that a gread wants
whole, in part, several to a piece and several pieces to a page, awaited by other blocks
meanwhile, and evicted soon after."""
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


def _file(datadir, size):
    path = os.path.join(datadir, "arriving_%d.bin" % size)
    np.random.default_rng(size).integers(0, 256, size, dtype=np.uint8).tofile(path)
    return path


@pytest.mark.parametrize("mode", ["MODE_ONDEMAND", "MODE_READAHEAD"])
@pytest.mark.parametrize("page,stride", [
    (32 * KiB, 128 * KiB), (32 * KiB, 160 * KiB), (64 * KiB, 16 * KiB), (64 * KiB, 200 * KiB + 8), (64 * KiB, 448 * KiB),
    (128 * KiB, 128 * KiB), (256 * KiB, 64 * KiB), (256 * KiB, 768 * KiB + 1), (512 * KiB, 512 * KiB), (1024 * KiB, 100 * KiB + 3),
])
def test_scans_of_whole_and_part_pages(torch_cuda, gfs, datadir, mode, page, stride):
    torch = torch_cuda
    size = max(24 * page, 12 * stride) + 1013
    pages = -(-size // page)
    path = _file(datadir, size)
    c, s, h = plain.scan_plain(path, stride)
    held = 12 * (-(-stride // page) + 1)  # pages that twelve greads touch at once
    for frames in (pages + 4, max(held, pages // 2)):
        with gfs.Context(cache_bytes=frames * page, page_size=page, mode=getattr(gfs, mode), max_rpc_pages=16) as ctx:
            fid = ctx.open(path)
            for again in range(3):
                cnt, sm, hs = ctx.scan(fid, stride, blocks=12, threads=(128, 256, 512)[again])
                torch.cuda.synchronize()
                assert cnt.cpu().numpy().tolist() == c
                assert np.array_equal(gfs.u64_view(sm), np.array(s, dtype=np.uint64))
                assert np.array_equal(gfs.u64_view(hs), np.array(h, dtype=np.uint64))
                st = ctx.stats()
                assert st["timeouts"] == 0
                if frames > pages and stride % page == 0:  # blocks that race for a page hold frames meanwhile
                    assert st["pages_fetched"] == pages and st["evictions"] == 0


@pytest.mark.parametrize("page,cols", [(64 * KiB, 1028), (64 * KiB, 8192), (256 * KiB, 1028), (256 * KiB, 12), (512 * KiB, 40000)])
def test_rows_come_out_the_same_while_they_arrive(torch_cuda, gfs, datadir, page, cols):
    """A row's sum has one order, whatever the pages and pieces: the first pass and one over
    cached pages give the same bits."""
    torch = torch_cuda
    rows = max(70, (5 << 20) // (4 * cols))
    m = (np.random.default_rng(cols).random((rows, cols), dtype=np.float32) * 2 - 1).astype(np.float32)
    path = os.path.join(datadir, "arriving_rows_%d.bin" % cols)
    m.tofile(path)
    vec = torch.from_numpy(np.random.default_rng(1).random(cols, dtype=np.float32)).cuda()
    with gfs.Context(cache_bytes=(4 * rows * cols // page + 8) * page, page_size=page, max_rpc_pages=16) as ctx:
        fid = ctx.open(path)
        read_len = max(1, (1 << 20) // (4 * cols)) * 4 * cols
        seen = []
        for _ in range(2):
            got = ctx.rowdot(fid, rows, cols, vec, stripe_rows=32, read_len=read_len, blocks=16)
            torch.cuda.synchronize()
            seen.append([v.cpu().numpy() for v in got])
        assert ctx.stats()["timeouts"] == 0
    for a, b in zip(*seen):
        assert np.array_equal(a, b)
    u = 2.0 ** -24  # |error| <= gamma_n * sum |a b|
    n = cols + 2
    bound = n * u / (1 - n * u) * (np.abs(m).astype(np.float64) @ vec.cpu().numpy().astype(np.float64))
    assert np.all(np.abs(seen[0][0] - m.astype(np.float64) @ vec.cpu().numpy().astype(np.float64)) <= bound)
    _, s, h = plain.scan_plain(path, 32 * cols * 4)
    assert np.array_equal(seen[0][1].view(np.uint64), np.array(s, dtype=np.uint64))
    assert np.array_equal(seen[0][2].view(np.uint64), np.array(h, dtype=np.uint64))
