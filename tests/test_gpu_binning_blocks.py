"""Binning of grids of 256 tiles and more, which are taken in blocks of at most 32
columns and rows together, or 64 on large grids: grid sizes around the switch and around the blocks' edges,
single rows and columns of tiles, Gaussian counts around a group, a batch of 1024 and
several batches per chunk (a tight capacity leaves few count rows), culled and
everything-covering Gaussians.  Lists are integers: bit-exact against the oracle's
(key, index) sort.  And the time: with footprints of a tile or two it follows the
lists, not Gaussians x tiles."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import oracle as ora
from paper_2505_05356_gb300 import gftorf

pytestmark = pytest.mark.gpu


def _case(seed, B, n, W, H, rmax):
    rng = np.random.default_rng(seed)
    u = rng.uniform(-10, W + 10, (B, n)).astype(np.float32)
    v = rng.uniform(-10, H + 10, (B, n)).astype(np.float32)
    r = rng.integers(1, rmax + 1, (B, n)).astype(np.int32)
    r[rng.random((B, n)) < 0.1] = 0                     # culled
    r[:, n // 2: n // 2 + 2] = max(W, H)                # nearly every tile
    r[1:, : n // 3] *= rng.random((max(B - 1, 0), n // 3)) < 0.3  # unequal visible counts
    z = rng.uniform(0.2, 6.0, (B, n)).astype(np.float32)
    z[:, ::7] = z[:, :1]                                # exact depth ties
    return u, v, r, z


def _compare(u, v, r, z, W, H, tile, tight):
    keys_o, vals_o, ranges_o = ora.bin_f32(u, v, r, z, W, H, *tile)
    dev = [torch.as_tensor(a, device="cuda") for a in (u, v, r, z)]
    cap = max(1, len(vals_o)) if tight else None
    keys, vals, ranges = gftorf.sort_footprints(*dev, W, H, tile, max_instances=cap)
    np.testing.assert_array_equal(ranges.cpu().numpy().astype(np.uint32).reshape(-1, 2),
                                  np.asarray(ranges_o, np.uint32).reshape(-1, 2))
    np.testing.assert_array_equal(keys.cpu().numpy().view(np.uint64), keys_o)
    np.testing.assert_array_equal(vals.cpu().numpy().astype(np.uint32), vals_o)


# 255, 256, 257, 511, 512 and more tiles, blocks with and without a remainder, one row and
# one column of tiles, one word per mask and two
@pytest.mark.parametrize("W,H,tile", [(120, 136, (8, 8)), (128, 128, (8, 8)), (2056, 8, (8, 8)),
                                      (584, 56, (8, 8)), (256, 128, (8, 8)),
                                      (8192, 16, (16, 16)), (16, 16000, (16, 16)),
                                      (517, 389, (16, 16)), (640, 480, (16, 16)),
                                      (496, 1000, (16, 32)), (1111, 777, (8, 8)),
                                      (4000, 2300, (64, 64))])
@pytest.mark.parametrize("B,n", [(1, 1), (1, 33), (3, 1023), (2, 1025), (1, 6000)])
@pytest.mark.parametrize("rmax", [3, 60])
def test_lists_bit_exact(W, H, tile, B, n, rmax):
    u, v, r, z = _case(W + 7 * H + n, B, n, W, H, rmax)
    _compare(u, v, r, z, W, H, tile, tight=False)


@pytest.mark.parametrize("W,H,tile,B,n", [(1500, 900, (8, 8), 1, 50000), (640, 480, (8, 8), 2, 3000),
                                          (1920, 1080, (16, 16), 3, 20000)])
def test_several_batches_per_chunk(W, H, tile, B, n):
    u, v, r, z = _case(n, B, n, W, H, 2)
    r[r > 2] = 0
    tiles = -(-W // tile[0]) * -(-H // tile[1])
    count = len(ora.bin_f32(u, v, r, z, W, H, *tile)[1])
    # rows of the counts: over the sort's buffers (3 words per Gaussian) or their own
    rows = max(3 * B * n // tiles, count // 8192 + 1 + B) + 1
    assert -(-n // (rows // B)) > 1024  # so a chunk is more than one batch
    _compare(u, v, r, z, W, H, tile, tight=True)


@pytest.mark.parametrize("W,H", [(640, 480), (1111, 777)])  # ranges by the scan, by their kernel
def test_overflow_leaves_empty_ranges_and_the_next_binning_whole(W, H):
    u, v, r, z = _case(5, 2, 3000, W, H, 20)
    keys_o, vals_o, ranges_o = ora.bin_f32(u, v, r, z, W, H, 8, 8)
    dev = [torch.as_tensor(a, device="cuda") for a in (u, v, r, z)]
    lib, tiles = gftorf.load(), -(-W // 8) * -(-H // 8)
    for cap, fits in ((len(vals_o) - 1, False), (len(vals_o), True)):
        d = gftorf.Dims(3000, 2, W, H, 8, 8, 1, 1, gftorf.F32, 0, 0, 0, 0, max_instances=cap)
        size = lib.gftorf_workspace_size(ctypes.byref(d))
        ws = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
        at = ws.data_ptr() + (-ws.data_ptr()) % 256
        vals = torch.empty(cap, dtype=torch.int32, device="cuda")
        ranges = torch.empty((2 * tiles, 2), dtype=torch.int32, device="cuda")
        count = torch.empty(1, dtype=torch.int64, device="cuda")
        for _ in range(2):  # the second finds what the first left behind
            assert lib.gftorf_sort_footprints(
                ctypes.byref(d), *(t.data_ptr() for t in dev), None, vals.data_ptr(),
                ranges.data_ptr(), count.data_ptr(), at, size,
                torch.cuda.current_stream().cuda_stream) == gftorf.OK
            n = ctypes.c_int64(0)
            code = lib.gftorf_read_device_status(ctypes.byref(d), at, size, ctypes.byref(n),
                                                 torch.cuda.current_stream().cuda_stream)
            assert n.value == len(vals_o) == count.item()
            assert code == (gftorf.OK if fits else gftorf.ERR_CAPACITY)
            if fits:
                np.testing.assert_array_equal(ranges.cpu().numpy().astype(np.uint32),
                                              np.asarray(ranges_o, np.uint32).reshape(-1, 2))
                np.testing.assert_array_equal(vals.cpu().numpy().astype(np.uint32), vals_o)
            else:
                assert not ranges.any().item()


def _bin_us(W, H, tile, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    u, v, z = (torch.rand((1, n), generator=g, device="cuda") * s + o
               for s, o in ((W, 0.0), (H, 0.0), (6.0, 0.2)))
    rad = torch.randint(1, 4, (1, n), generator=g, device="cuda", dtype=torch.int32)
    _, vals, ranges = gftorf.sort_footprints(u, v, rad, z, W, H, tile)
    lib, m = gftorf.load(), vals.numel()
    d = gftorf.Dims(n, 1, W, H, *tile, 1, 1, gftorf.F32, 0, 0, 0, 0, max_instances=m)
    size = lib.gftorf_workspace_size(ctypes.byref(d))
    ws = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
    at = ws.data_ptr() + (-ws.data_ptr()) % 256
    count = torch.empty(1, dtype=torch.int64, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    assert lib.gftorf_sort_footprints(ctypes.byref(d), u.data_ptr(), v.data_ptr(), rad.data_ptr(),
                                      z.data_ptr(), None, vals.data_ptr(), ranges.data_ptr(),
                                      count.data_ptr(), at, size, stream) == gftorf.OK
    times = []
    for i in range(15):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        assert lib.gftorf_bin(ctypes.byref(d), at, size, stream) == gftorf.OK
        e1.record()
        e1.synchronize()
        if i >= 4:
            times.append(e0.elapsed_time(e1) * 1e3)
    return sorted(times)[len(times) // 2], m


def test_time_follows_the_lists():
    """300k Gaussians of radius 1 to 3 on 1200 and on 32400 tiles of 16x16: lists of the
    same length.  Work per (group of Gaussians, tile) would cost 27 times as much."""
    small, m0 = _bin_us(640, 480, (16, 16), 300_000)
    large, m1 = _bin_us(3840, 2160, (16, 16), 300_000)
    assert 0.9 < m1 / m0 < 1.1
    assert large <= 8 * small, (small, large)
