"""Read lengths far beyond the file and beyond 32 bits: nothing is allocated for them, so they
have to be served like one read of the whole, with a reserve that does not wrap around."""
import os
import time

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


@pytest.mark.parametrize("read_len,stripe", [(64 << 32, 7), (64 * ((1 << 32) + 3), 40), (64 << 45, (1 << 32) - 1), (64 * 5, (1 << 32) - 1)])
def test_rowdot_pieces_longer_than_32_bits_of_rows(torch_cuda, gfs, datadir, read_len, stripe):
    torch = torch_cuda
    rows, cols = 50, 16
    m = np.random.default_rng(61).integers(-8, 8, (rows, cols)).astype(np.float32)
    path = os.path.join(datadir, "huge_rows.f32")
    m.tofile(path)
    vec = torch.arange(cols, dtype=torch.float32, device="cuda")
    with gfs.Context(cache_bytes=64 * 4 * KiB, page_size=4 * KiB, timeout_ns=2_000_000_000) as ctx:
        fid = ctx.open(path)
        out, ssum, shash, status = ctx.rowdot(fid, rows, cols, vec, stripe_rows=stripe, read_len=read_len, blocks=8)
        torch.cuda.synchronize()
        assert status.item() == 0
        assert np.array_equal(out.cpu().numpy(), m @ np.arange(cols, dtype=np.float32))  # exact in float32
        _, s, h = plain.scan_plain(path, min(stripe, rows) * cols * 4)
        assert np.array_equal(gfs.u64_view(ssum), np.array(s, dtype=np.uint64))
        assert np.array_equal(gfs.u64_view(shash), np.array(h, dtype=np.uint64))


@pytest.mark.parametrize("read_len", [1 << 40, (1 << 64) - 16])
def test_histogram_piece_of_any_length(torch_cuda, gfs, datadir, read_len):
    torch = torch_cuda
    v = np.random.default_rng(62).integers(0, 9000, 30000, dtype=np.int32)
    path = os.path.join(datadir, "huge_hist.i32")
    v.tofile(path)
    with gfs.Context(cache_bytes=64 * 4 * KiB, page_size=4 * KiB) as ctx:
        fid = ctx.open(path)
        hist, sums, status = ctx.histogram(fid, nbins=9000, read_len=read_len, blocks=8)
        torch.cuda.synchronize()
        assert status.item() == 0
        assert np.array_equal(hist.cpu().numpy(), np.bincount(v, minlength=9000))


def test_reserve_of_a_huge_product_leaves_readahead_no_frame(torch_cuda, gfs, datadir):
    """65536 blocks of 65536 pages are 2^32 pages: all frames stay reserved, not one."""
    torch = torch_cuda
    page = 4 * KiB
    v = np.random.default_rng(63).integers(0, 9000, 64 * page // 4, dtype=np.int32)
    path = os.path.join(datadir, "huge_reserve.i32")
    v.tofile(path)
    with gfs.Context(cache_bytes=256 * page, page_size=page) as ctx:
        fid = ctx.open(path)
        hist, _, status = ctx.histogram(fid, nbins=9000, read_len=65536 * page, blocks=65536)
        torch.cuda.synchronize()
        st = ctx.stats()
        assert status.item() == 0 and np.array_equal(hist.cpu().numpy(), np.bincount(v, minlength=9000))
        assert st["ra_pages_sync"] == st["ra_pages_async"] == 0


@pytest.mark.parametrize("unit", [1 << 40, (1 << 64) - 1])
def test_serving_units_of_any_length(torch_cuda, gfs, datadir, unit):
    path = os.path.join(datadir, "huge_unit.bin")
    data = np.random.default_rng(64).integers(0, 256, 200_001, dtype=np.uint8)
    data.tofile(path)
    with gfs.Context(cache_bytes=256 * 4 * KiB, page_size=4 * KiB) as ctx:
        fid = ctx.open(path)
        ctx.serve_start(ctas=16, threads=256, unit_bytes=unit, max_requests=4, queue_slots=4)
        try:
            assert ctx.submit_scan(fid, 0, len(data), 5)
            done, late = [], time.monotonic() + 20
            while not done and time.monotonic() < late:
                done = ctx.poll()
        finally:
            ctx.serve_stop()
    assert done[0]["tag"] == 5 and done[0]["status"] == 0 and done[0]["bytes"] == len(data)
    assert done[0]["sum"] == plain.byte_sum(data.tobytes()) and done[0]["hash"] == plain.pos_hash(data.tobytes(), 0)
