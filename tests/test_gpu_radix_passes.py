"""The radix passes of bin/sort at item counts around their tile sizes, the
groups of tiles their look-back works in and the sizes at which the tile size
changes: one instance per splat, against numpy's stable sort by tile and depth,
with the count read back and without synchronising (passes sized by a larger
capacity)."""
import numpy as np
import pytest
import torch

from paper_2604_02120_gb300 import gs

pytestmark = pytest.mark.gpu

TILES_X, TILES_Y = 1200, 4  # 300 supertiles: two digits, the second of one bit


@pytest.mark.parametrize("n", [1, 31, 1023, 1025, 8192, 8193, 262144, 262145, 16384 * 17 + 5, 9 << 17, (9 << 17) + 1,
                               32768 * 40 + 4097])
def test_one_instance_per_splat_sorts_stably(n):
    rng = np.random.default_rng(n)
    tile = rng.integers(0, TILES_X * TILES_Y, n)
    mean = np.stack([tile % TILES_X * 16 + 8, tile // TILES_X * 16 + 8], 1).astype(np.float32)
    # few exponents, many ties, all four digits in use
    depth = rng.choice(rng.uniform(0.2, 300.0, max(1, n // 2)).astype(np.float32), n)
    want = np.lexsort((np.arange(n), depth, tile))
    m, d = torch.from_numpy(mean).cuda(), torch.from_numpy(depth).cuda()
    r = torch.ones(n, dtype=torch.int32, device="cuda")
    w, h = TILES_X * 16, TILES_Y * 16
    for cap, graph in ((n, False), (n, True), (3 * n + 5000, True)):
        ws = torch.full((gs.gs_bin_sort_workspace_size(n, cap, w, h) + 256,), 255, device="cuda", dtype=torch.uint8)
        ids = torch.full((cap,), -1, device="cuda", dtype=torch.int32)
        ranges = torch.zeros(2 * gs.num_tiles(w, h), device="cuda", dtype=torch.int32)
        cnt = torch.zeros(1, device="cuda", dtype=torch.int64)
        for _ in range(2):  # the second time on the workspace the first one left
            gs.gs_bin_sort_views(1, n, m, r, d, [w], [h], cap, ws, None, ids, ranges, count_dev=cnt if graph else None)
            assert gs.gs_sync_status() == gs.GS_OK
            np.testing.assert_array_equal(ids[:n].cpu().numpy(), want)
        if graph:
            assert int(cnt) == n
