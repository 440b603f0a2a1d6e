"""Runs of cached pages that every warp of a block looks up, cut at every kind of gap.
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


def _bytes_file(datadir, size, seed):
    path = os.path.join(datadir, "sinks_%d_%d.bin" % (size, seed))
    np.random.default_rng(seed).integers(0, 256, size, dtype=np.uint8).tofile(path)
    return path


@pytest.mark.parametrize("page,threads", [(4 * KiB, 128), (4 * KiB, 512), (16 * KiB, 256)])
def test_runs_of_many_warps_stop_at_every_gap(torch_cuda, gfs, datadir, page, threads):
    """Greads over a cache that holds scattered pages: runs end at pages 1, 31, 32, 33, ... ."""
    torch = torch_cuda
    pages = 20 * threads // 32
    size = pages * page - 77
    path = _bytes_file(datadir, size, 24)
    ref = np.fromfile(path, dtype=np.uint8)
    t = lambda v: torch.tensor(v, dtype=torch.int64, device="cuda")  # noqa: E731
    for holes in ([0], [1], [31], [32], [33], [63, 64], list(range(5, pages, 37)), [pages - 1]):
        holes = [h for h in holes if h < pages]
        with gfs.Context(cache_bytes=2 * pages * page, page_size=page) as ctx:
            fid = ctx.open(path)
            ctx.fadvise(fid, gfs.ADV_RANDOM)
            keep = [p for p in range(pages) if p not in holes]
            buf = torch.zeros(pages * page, dtype=torch.uint8, device="cuda")
            ret = torch.zeros(len(keep), dtype=torch.int64, device="cuda")
            ctx.read_many(fid, t([p * page for p in keep]), t([page] * len(keep)), t([p * page for p in keep]), buf, ret,
                          blocks=8, threads=128)
            torch.cuda.synchronize()
            before = ctx.stats()
            buf = torch.zeros(size + 32, dtype=torch.uint8, device="cuda")
            ret = torch.zeros(1, dtype=torch.int64, device="cuda")
            ctx.read_many(fid, t([3]), t([size]), t([5]), buf, ret, blocks=1, threads=threads)
            torch.cuda.synchronize()
            st = ctx.stats()
            assert ret.item() == size - 3
            assert np.array_equal(buf.cpu().numpy()[5:5 + size - 3], ref[3:])
            assert st["hits"] - before["hits"] == len(keep)
            assert st["misses"] - before["misses"] == len(holes)
            assert st["evictions"] == 0
