"""The per-tile sort at the edges of its forms (one warp up to 256, 512 and 1024
entries, a CTA up to 4096), on depths that its 32-bit keys separate, round
together or cannot tell apart: (tile, depth, id) order bit for bit against
numpy, through gs_bin_tiles."""
import numpy as np
import pytest
import torch

from tests._util import ensure_built

pytestmark = pytest.mark.gpu

LENGTHS = (1, 2, 7, 8, 9, 31, 32, 33, 128, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 1500, 2047, 2048, 2049, 3000,
           4095, 4096)


def _depths(kind, rng, n):
    one = np.float32(1.5).view(np.uint32)
    if kind == "spread":
        return rng.uniform(0.5, 6.0, n).astype(np.float32)
    if kind == "wide":
        return np.exp(rng.uniform(np.log(0.21), np.log(1e6), n)).astype(np.float32)
    if kind == "ulps":  # neighbouring float values: many equal ones
        return (one + rng.integers(0, max(2, n // 3), n).astype(np.uint32)).view(np.float32)
    if kind == "pairs":  # every value twice, one far outlier that coarsens the rounding
        d = np.repeat(rng.uniform(1.0, 2.0, (n + 1) // 2).astype(np.float32), 2)[:n]
        d[0] = 1e5
        return rng.permutation(d)
    if kind == "few":  # a handful of equal values in a spread list
        d = rng.uniform(0.5, 6.0, n).astype(np.float32)
        k = min(n, 5)
        d[rng.choice(n, k, replace=False)] = d[0]
        return d
    if kind == "runs":  # one run longer than the run limit
        d = rng.uniform(0.5, 6.0, n).astype(np.float32)
        d[rng.choice(n, min(n, 40), replace=False)] = np.float32(2.0)
        return d
    return np.full(n, 1.25, np.float32)  # equal


@pytest.mark.parametrize("kind", ["spread", "wide", "ulps", "pairs", "few", "runs", "equal"])
def test_lists_of_every_form(kind):
    ensure_built()
    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context
    rng = np.random.default_rng(5)
    order = rng.permutation(len(LENGTHS))  # forms mixed within a CTA
    tile = np.concatenate([np.full(LENGTHS[k], t) for t, k in enumerate(order)])
    depth = np.concatenate([_depths(kind, rng, LENGTHS[k]) for k in order])
    mix = rng.permutation(tile.size)
    tile, depth = tile[mix], depth[mix]
    W, H = 16 * len(LENGTHS), 16
    mean = np.stack([16.0 * tile + rng.uniform(4, 12, tile.size), rng.uniform(4, 12, tile.size)], 1).astype(np.float32)
    ext = np.full((tile.size, 2), 1.0, np.float32)
    ctx = Context(0)
    cu = lambda a: torch.as_tensor(a, device="cuda")
    keys = torch.empty(tile.size, dtype=torch.int64, device="cuda")
    ids = torch.empty(tile.size, dtype=torch.int32, device="cuda")
    ranges = torch.empty((len(LENGTHS), 2), dtype=torch.int32, device="cuda")
    n = abi.gs_bin_tiles(ctx.handle, cu(mean), cu(ext), cu(depth), W, H, 16, 16, keys, ids, ranges)
    assert n == tile.size
    want = np.lexsort((np.arange(tile.size), depth, tile))
    assert np.array_equal(ids.cpu().numpy(), want)
    k64 = (tile[want].astype(np.uint64) << np.uint64(32)) | depth[want].view(np.uint32).astype(np.uint64)
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), k64)
    lens = (ranges[:, 1] - ranges[:, 0]).cpu().numpy()
    assert np.array_equal(lens, np.array(LENGTHS)[order])
    ctx.close()
