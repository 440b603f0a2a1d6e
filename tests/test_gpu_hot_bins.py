"""Histograms whose hot values lie above the bins that are kept in shared memory: counted
once a value or once a warp, the counts are the same."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
KiB = 1024
SMEM = 8192  # bins kept in shared memory


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


def _values(kind, n):
    rng = np.random.default_rng(41)
    wide = rng.integers(0, 1 << 17, n)
    return {
        "one": lambda: np.full(n, 50000),
        "half": lambda: np.where(rng.random(n) < 0.5, 50000, wide),
        "tenth": lambda: np.where(rng.random(n) < 0.1, SMEM, wide),
        "edges": lambda: rng.choice([0, SMEM - 1, SMEM, SMEM + 1, (1 << 17) - 1], n),
        "few": lambda: rng.integers(SMEM, SMEM + 64, n),
        "sorted": lambda: np.sort(wide),
        "patches": lambda: np.where(np.arange(n) // 700 % 3 == 0, 60000, wide),  # hot and cold units in turn
        "negative": lambda: np.where(rng.random(n) < 0.3, -1, wide),
    }[kind]().astype(np.int32)


@pytest.mark.parametrize("kind", ["one", "half", "tenth", "edges", "few", "sorted", "patches", "negative"])
def test_hot_high_bins_are_counted_exactly(torch_cuda, gfs, datadir, kind):
    torch = torch_cuda
    n = 600_001  # the last piece and its last unit are short
    v = _values(kind, n)
    path = os.path.join(datadir, "hot_bins.i32")
    v.tofile(path)
    u = v.view(np.uint32)
    for nbins in (1 << 17, 50001, SMEM + 1):
        want = np.bincount(u[u < nbins], minlength=nbins)
        with gfs.Context(cache_bytes=4096 * KiB, page_size=64 * KiB) as ctx:
            fid = ctx.open(path)
            for read_len in (256 * KiB, 48 * KiB):
                hist, sums, status = ctx.histogram(fid, nbins=nbins, read_len=read_len, blocks=8)
                torch.cuda.synchronize()
                assert status.item() == 0
                assert np.array_equal(hist.cpu().numpy(), want)
                assert int(gfs.u64_view(sums)[1]) == int((u >= nbins).sum())
