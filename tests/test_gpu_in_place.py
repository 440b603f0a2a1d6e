"""Row dot products and histograms taken where their pages lie: rows and pieces that pages cut anywhere.
"""
import os

import numpy as np
import pytest

from oracle import apps, plain

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


@pytest.mark.parametrize("rows,cols,rows_read,page,frames", [
    (37, 1028, 3, 4 * KiB, 64),       # rows a little longer than a page
    (37, 1028, 37, 4 * KiB, 512),     # one gread of more pages than a warp looks up
    (19, 20004, 2, 64 * KiB, 16),     # rows longer than a page
    (9, 20004, 3, 4 * KiB, 128),      # rows of twenty pages
    (515, 4, 64, 4 * KiB, 16),        # rows of one word
    (130, 132, 130, 16 * KiB, 16),    # rows of 33 words
    (64, 8192, 32, 512 * KiB, 8),
])
def test_rowdot_rows_across_pages(torch_cuda, gfs, datadir, rows, cols, rows_read, page, frames):
    torch = torch_cuda
    rng = np.random.default_rng(25)
    mat = (rng.random((rows, cols), dtype=np.float32) * 2 - 1).astype(np.float32)
    vec = (rng.random(cols, dtype=np.float32) * 2 - 1).astype(np.float32)
    path = os.path.join(datadir, "sinks_mat.f32")
    mat.tofile(path)
    ref, ab = apps.rowdot(path, rows, cols, vec)
    stripe = max(1, rows // 3)
    data = mat.tobytes()
    outs = []
    with gfs.Context(cache_bytes=frames * page, page_size=page) as ctx:
        fid = ctx.open(path)
        for _ in range(2):
            out, ssum, shash, status = ctx.rowdot(fid, rows, cols, torch.from_numpy(vec).cuda(), stripe,
                                                  rows_read * cols * 4, blocks=2)
            torch.cuda.synchronize()
            assert status.item() == 0
            outs.append(out.cpu().numpy())
            assert np.all(np.abs(outs[-1].astype(np.float64) - ref) <= apps.gamma(cols) * ab)
            for s in range(len(ssum)):
                o = s * stripe * cols * 4
                part = data[o:o + stripe * cols * 4]
                assert int(gfs.u64_view(ssum)[s]) == plain.byte_sum(part)
                assert int(gfs.u64_view(shash)[s]) == plain.pos_hash(part, o)
    assert np.array_equal(outs[0], outs[1])  # one order of additions, wherever runs end


@pytest.mark.parametrize("extra", [0, 1, 4, 7, 12])
@pytest.mark.parametrize("page,read_len", [(4 * KiB, 48), (4 * KiB, 80 * KiB), (64 * KiB, 96 * KiB + 16)])
def test_histogram_ends_at_any_byte(torch_cuda, gfs, datadir, extra, page, read_len):
    torch = torch_cuda
    rng = np.random.default_rng(26)
    vals = rng.integers(0, 20000, 50000 if read_len > 48 else 900, dtype=np.int32)
    data = vals.tobytes()[:len(vals) * 4 - 16] + rng.integers(0, 3, extra, dtype=np.uint8).tobytes()
    path = os.path.join(datadir, "sinks_hist.i32")
    with open(path, "wb") as f:
        f.write(data)
    whole = np.frombuffer(data[:len(data) // 4 * 4], dtype=np.uint32)
    for nbins in (20000, 300):
        want = np.bincount(whole[whole < nbins], minlength=nbins)
        with gfs.Context(cache_bytes=512 * KiB, page_size=page) as ctx:
            fid = ctx.open(path)
            for _ in range(2):
                hist, sums, status = ctx.histogram(fid, nbins=nbins, read_len=read_len, blocks=4)
                torch.cuda.synchronize()
                assert status.item() == 0
                assert np.array_equal(hist.cpu().numpy(), want)
                assert gfs.u64_view(sums).tolist() == [plain.byte_sum(data), int((whole >= nbins).sum())]
