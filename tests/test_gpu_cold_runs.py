"""Greads over caches that hold some of their pages: after a miss of one page no run is
looked for at the next, and a page that a look-up did not find is not looked up again.  The
delivered bytes and the counters have to be those of pages taken one by one."""
import os

import numpy as np
import pytest

from oracle import plain

pytestmark = pytest.mark.gpu
KiB = 1024
PAGES, STRIDE = 43, 9  # pages of the file (the last one short), pages of a gread


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


def _held():
    """Sets of cached pages: none, all, every second, runs of two and three, the ends of greads."""
    every = range(PAGES)
    yield []
    yield list(every)
    yield [p for p in every if p % 2]
    yield [p for p in every if p % 5 in (1, 2)]
    yield [p for p in every if p % 7 < 3]
    yield [p for p in every if p % STRIDE == 0]
    yield [p for p in every if p % STRIDE == STRIDE - 1]


@pytest.mark.parametrize("xfer", [1, 2])
@pytest.mark.parametrize("page,threads", [(4 * KiB, 128), (16 * KiB, 256), (64 * KiB, 512), (256 * KiB, 256)])
def test_on_demand_scans_count_each_page_once(torch_cuda, gfs, datadir, xfer, page, threads):
    torch = torch_cuda
    size = PAGES * page - 333
    path = os.path.join(datadir, "cold_runs_%d.bin" % page)
    np.random.default_rng(31).integers(0, 256, size, dtype=np.uint8).tofile(path)
    c, s, h = plain.scan_plain(path, STRIDE * page)
    t = lambda v: torch.tensor(v, dtype=torch.int64, device="cuda")  # noqa: E731
    for held in _held():
        with gfs.Context(cache_bytes=2 * PAGES * page, page_size=page, mode=gfs.MODE_ONDEMAND, xfer=xfer) as ctx:
            fid = ctx.open(path)
            if held:
                buf = torch.zeros(16 * len(held), dtype=torch.uint8, device="cuda")
                ctx.read_many(fid, t([p * page for p in held]), t([16] * len(held)), t([16 * i for i in range(len(held))]),
                              buf, torch.zeros(len(held), dtype=torch.int64, device="cuda"), blocks=4, threads=128)
                torch.cuda.synchronize()
            before = ctx.stats()
            cnt, sm, hs = ctx.scan(fid, STRIDE * page, blocks=3, threads=threads)
            torch.cuda.synchronize()
            st = ctx.stats()
            assert cnt.cpu().numpy().tolist() == c
            assert np.array_equal(gfs.u64_view(sm), np.array(s, dtype=np.uint64))
            assert np.array_equal(gfs.u64_view(hs), np.array(h, dtype=np.uint64))
            assert st["hits"] - before["hits"] == len(held)
            assert st["misses"] - before["misses"] == PAGES - len(held)
            assert st["evictions"] == st["retries"] == st["timeouts"] == 0
