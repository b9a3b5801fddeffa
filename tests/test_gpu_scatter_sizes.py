"""The scatter of pairs into tile lists (64 or 256 items per block by the number
of items, large rectangles from the queue) against numpy, at the edges of its
rounds and of the rule."""
import numpy as np
import pytest
import torch

from tests._util import ensure_built

pytestmark = pytest.mark.gpu


def _scatter_limit():  # items up to which a block takes 64 of them
    return 64 * 16 * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("n", [1, 63, 64, 65, 257, "limit", "limit + 1"])
def test_scatter_sizes(n):
    ensure_built()
    from paper_2408_12677_gb300 import abi
    from paper_2408_12677_gb300.torch_api import Context
    n = {"limit": _scatter_limit(), "limit + 1": _scatter_limit() + 1}.get(n, n)
    rng = np.random.default_rng(n)
    TX, TY = 65, 50  # lists stay below the per-tile sort's longest
    tx, ty = rng.integers(0, TX, n), rng.integers(0, TY, n)
    k = np.zeros((n, 2), np.int64)  # tiles on each side of the centre's
    big = rng.permutation(n)[:max(1, min(n // 8, 300))]
    k[big] = rng.integers(0, 12, (big.size, 2))
    mean = (16.0 * np.stack([tx, ty], 1) + 8.0).astype(np.float32)
    depth = rng.uniform(0.5, 6.0, n).astype(np.float32)
    item, tile = [], []
    for i in range(n) if n < 1000 else big:
        x = np.arange(max(tx[i] - k[i, 0], 0), min(tx[i] + k[i, 0], TX - 1) + 1)
        y = np.arange(max(ty[i] - k[i, 1], 0), min(ty[i] + k[i, 1], TY - 1) + 1)
        t = (y[:, None] * TX + x[None]).ravel()
        item.append(np.full(t.size, i))
        tile.append(t)
    if n >= 1000:
        rest = np.setdiff1d(np.arange(n), big)
        item.append(rest)
        tile.append((ty * TX + tx)[rest])
    item, tile = np.concatenate(item), np.concatenate(tile)
    want = np.lexsort((item, depth[item], tile))
    ctx = Context(0)
    cu = lambda a: torch.as_tensor(a, device="cuda")
    keys = torch.empty(tile.size, dtype=torch.int64, device="cuda")
    ids = torch.empty(tile.size, dtype=torch.int32, device="cuda")
    ranges = torch.empty((TX * TY, 2), dtype=torch.int32, device="cuda")
    got = abi.gs_bin_tiles(ctx.handle, cu(mean), cu((16.0 * k + 1.0).astype(np.float32)), cu(depth), 16 * TX, 16 * TY, 16,
                           16, keys, ids, ranges)
    assert got == tile.size
    assert np.array_equal(ids.cpu().numpy(), item[want])
    lens = (ranges[:, 1] - ranges[:, 0]).cpu().numpy()
    assert np.array_equal(lens, np.bincount(tile, minlength=TX * TY))
    ctx.close()
