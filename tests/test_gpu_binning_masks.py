"""The tile-mask binning at its edges: columns + rows of tiles just below, at and
above the 32-bit words of the masks (one to several words), Gaussian counts
around a group of 32, a chunk and a sort tile, rectangles that cover one tile,
whole rows, whole columns or everything, several frames with unequal visible
counts.  Lists are integers: bit-exact against the oracle's (key, index) sort."""
import numpy as np
import pytest
import torch

from oracle import oracle as ora
from paper_2505_05356_gb300 import gftorf

pytestmark = pytest.mark.gpu


def _case(seed, B, n, W, H):
    rng = np.random.default_rng(seed)
    u = rng.uniform(-20, W + 20, (B, n)).astype(np.float32)
    v = rng.uniform(-20, H + 20, (B, n)).astype(np.float32)
    r = rng.integers(1, 40, (B, n)).astype(np.int32)
    kind = rng.integers(0, 100, (B, n))
    r[kind < 10] = 1
    r[(kind == 10) | (np.arange(n) == 7)] = max(W, H)  # covers nearly every tile
    r[kind > 90] = 0                                   # culled
    r[:, : n // 3] *= (rng.random((B, n // 3)) < 0.5)  # unequal visible counts
    z = rng.uniform(0.2, 6.0, (B, n)).astype(np.float32)
    z[:, ::5] = z[:, :1]                  # exact depth ties
    return u, v, r, z


@pytest.mark.parametrize("W,H,tile", [(8, 8, (8, 8)), (120, 128, (8, 8)), (128, 128, (8, 8)),
                                      (136, 128, (8, 8)), (250, 260, (8, 8)), (517, 389, (16, 16)),
                                      (1024, 17, (16, 16)), (16, 1000, (16, 32)),
                                      (640, 480, (32, 32)), (640, 576, (64, 64)),
                                      (1500, 900, (8, 8))])
@pytest.mark.parametrize("B,n", [(1, 1), (1, 31), (2, 33), (3, 257), (2, 5000)])
def test_lists_bit_exact(W, H, tile, B, n):
    u, v, r, z = _case(W * 31 + H + n, B, n, W, H)
    keys_o, vals_o, ranges_o = ora.bin_f32(u, v, r, z, W, H, tile[0], tile[1])
    dev = [torch.as_tensor(a, device="cuda") for a in (u, v, r, z)]
    keys, vals, ranges = gftorf.sort_footprints(*dev, W, H, tile)
    np.testing.assert_array_equal(ranges.cpu().numpy().astype(np.uint32).reshape(-1, 2),
                                  np.asarray(ranges_o, np.uint32).reshape(-1, 2))
    np.testing.assert_array_equal(keys.cpu().numpy().view(np.uint64), keys_o)
    np.testing.assert_array_equal(vals.cpu().numpy().astype(np.uint32), vals_o)
