"""The duplication of full rectangles works in tiles of 256 items up to 65536 items
and of 1024 beyond: lists of splats that cover one to hundreds of supertiles, at
counts around a tile and around that line, against a stable sort in numpy."""
import numpy as np
import pytest
import torch

from paper_2604_02120_gb300 import gs

pytestmark = pytest.mark.gpu
W, H = 1000, 300  # 63 x 19 tiles, 16 x 5 supertiles


def _expected(mean, radius, depth):
    tx, ty = (W + 15) // 16, (H + 15) // 16
    f, r = np.floor(mean).astype(np.int64), radius.astype(np.int64)
    x0, x1 = np.maximum((f[:, 0] - r) // 16, 0), np.minimum((f[:, 0] + r) // 16, tx - 1)
    y0, y1 = np.maximum((f[:, 1] - r) // 16, 0), np.minimum((f[:, 1] + r) // 16, ty - 1)
    w = np.where(r > 0, np.maximum(x1 - x0 + 1, 0), 0)
    cnt = w * np.maximum(y1 - y0 + 1, 0)
    g = np.repeat(np.arange(len(r)), cnt)
    j = np.arange(cnt.sum()) - np.repeat(np.cumsum(cnt) - cnt, cnt)
    tile = (y0[g] + j // w[g]) * tx + x0[g] + j % w[g]
    o = np.lexsort((g, depth[g], tile))
    return g[o], np.bincount(tile, minlength=tx * ty)


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1025, 65535, 65536, 65537, 66561])
def test_rectangles_of_many_supertiles(n):
    rng = np.random.default_rng(n)
    mean = rng.uniform([-40, -40], [W + 40, H + 40], (n, 2)).astype(np.float32)
    radius = rng.integers(0, 40, n).astype(np.int32)
    big = rng.random(n) < min(1.0, 300 / n)
    radius[big] = rng.integers(100, 1500, big.sum())
    depth = rng.choice(rng.uniform(0.2, 9.0, max(1, n // 2)).astype(np.float32), n)
    ids, per = _expected(mean, radius, depth)
    m, r, d = (torch.from_numpy(a).cuda() for a in (mean, radius, depth))
    nt, cap = gs.num_tiles(W, H), max(len(ids), 1)
    ws = torch.full((gs.gs_bin_sort_workspace_size(n, cap, W, H) + 256,), 255, device="cuda", dtype=torch.uint8)
    cnt = torch.zeros(1, device="cuda", dtype=torch.int64)
    for graph in (False, True):
        out = torch.full((cap + 64,), -1, device="cuda", dtype=torch.int32)
        ranges = torch.zeros(2 * nt, device="cuda", dtype=torch.int32)
        _, count = gs.gs_bin_sort_views(1, n, m, r, d, [W], [H], cap, ws, None, out, ranges,
                                        count_dev=cnt if graph else None)
        assert gs.gs_sync_status() == gs.GS_OK and (int(cnt) if graph else count) == len(ids)
        np.testing.assert_array_equal(out[:len(ids)].cpu().numpy(), ids)
        assert (out[cap:] == -1).all()
        got = ranges.cpu().numpy().reshape(-1, 2)
        np.testing.assert_array_equal(got[:, 1] - got[:, 0], per)
    if len(ids) > 3:  # cut off
        small = len(ids) * 2 // 3
        out = torch.full((cap + 64,), -1, device="cuda", dtype=torch.int32)
        gs.gs_bin_sort_views(1, n, m, r, d, [W], [H], small, ws, None, out, ranges, count_dev=cnt)
        assert gs.gs_sync_status() == gs.GS_ERR_CAPACITY and int(cnt) == len(ids)
        assert (out[small:] == -1).all() and int(ranges.max()) <= small
