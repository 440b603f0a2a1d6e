"""Copy-out at every phase: source and buffer each start at any byte of a 16-byte word.

The copy stores 16 bytes a thread after a head of single bytes; where the source sits at
another phase it shifts two aligned words together.  Lengths cover the edges of the head,
the body (one lane, one warp, one pass of a block) and the tail, inside one page, across a
page end and at the end of the file.  Bytes around each destination must stay as they were.
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


@pytest.mark.parametrize("page,threads", [(4 * KiB, 128), (64 * KiB, 256), (64 * KiB, 512)])
def test_reads_at_every_phase(torch_cuda, gfs, datadir, page, threads):
    torch = torch_cuda
    size = 3 * 64 * KiB + 4099
    ref = np.random.default_rng(5).integers(0, 256, size, dtype=np.uint8)
    path = os.path.join(datadir, "phases.bin")
    ref.tofile(path)
    lens = [1, 2, 15, 16, 17, 31, 33, 511, 512, 513, 527, 2047, 4096, 4097, 8205, 3 * page + 5]
    offs, dsts, ns, pos = [], [], [], 64
    for i, n in enumerate(lens):
        for k in range(16):
            base = [0, page - n // 2 - 8, size - n - 15][(i + k) % 3]
            offs.append(max(base, 0) + k)
            dsts.append(pos + (5 * k + i) % 16)
            ns.append(n)
            pos += n + 64
    want = np.full(pos + 64, 0xA5, dtype=np.uint8)
    for o, d, n in zip(offs, dsts, ns):
        part = ref[o:o + n]
        want[d:d + len(part)] = part
    t = lambda v: torch.tensor(v, dtype=torch.int64, device="cuda")  # noqa: E731
    with gfs.Context(cache_bytes=512 * KiB, page_size=page) as ctx:
        fid = ctx.open(path)
        for _ in range(2):  # from the file, then from the cache
            buf = torch.full((len(want),), 0xA5, dtype=torch.uint8, device="cuda")
            ret = torch.zeros(len(offs), dtype=torch.int64, device="cuda")
            ctx.read_many(fid, t(offs), t(ns), t(dsts), buf, ret, blocks=12, threads=threads)
            torch.cuda.synchronize()
            assert ret.cpu().tolist() == [min(n, size - o) for o, n in zip(offs, ns)]
            assert np.array_equal(buf.cpu().numpy(), want)


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("stride", [65521, 96 * KiB + 8, 4095])
def test_scan_strides_at_every_phase(torch_cuda, gfs, datadir, stride, fused):
    from oracle import plain
    size = 1234567
    ref = np.random.default_rng(6).integers(0, 256, size, dtype=np.uint8)
    path = os.path.join(datadir, "strides.bin")
    ref.tofile(path)
    want = plain.scan_plain(path, stride)
    for page in (4 * KiB, 64 * KiB):
        with gfs.Context(cache_bytes=4 << 20, page_size=page) as ctx:
            fid = ctx.open(path)
            for _ in range(2):
                cnt, sm, hs = ctx.scan_host(fid, stride, blocks=16, fused=fused)
                assert (cnt.tolist(), sm.tolist(), hs.tolist()) == tuple(list(w) for w in want)
