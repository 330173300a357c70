"""The per-tile lists of one supertile (64 x 64 pixels and ragged images around it)
at pair counts around the rounds of 512 and the batches of 128 the last bin/sort
kernels work in, against a stable sort in numpy: with keys and the count read back,
without keys and without synchronising, and cut off at the capacity."""
import numpy as np
import pytest
import torch

from paper_2604_02120_gb300 import gs

pytestmark = pytest.mark.gpu


def _items(n, width, height, seed):
    rng = np.random.default_rng(seed)
    mean = rng.uniform([-8, -8], [width + 8, height + 8], (n, 2)).astype(np.float32)
    radius = rng.integers(0, 40, n).astype(np.int32)
    depth = rng.choice(np.linspace(0.5, 3.0, max(2, n // 3)), n).astype(np.float32)  # with ties
    return mean, radius, depth


def _expected(mean, radius, depth, width, height):
    tx, ty = (width + 15) // 16, (height + 15) // 16
    keys, ids = [], []
    f = np.floor(mean).astype(np.int64)
    for g in range(len(radius)):
        r = int(radius[g])
        if r <= 0:
            continue
        x0, x1 = max((f[g, 0] - r) // 16, 0), min((f[g, 0] + r) // 16, tx - 1)
        y0, y1 = max((f[g, 1] - r) // 16, 0), min((f[g, 1] + r) // 16, ty - 1)
        bits = int(depth[g:g + 1].view(np.uint32)[0])
        for y in range(y0, y1 + 1):
            for x in range(x0, x1 + 1):
                keys.append(((y * tx + x) << 32) | bits)
                ids.append(g)
    keys, ids = np.array(keys, np.uint64), np.array(ids, np.int64)
    o = np.argsort(keys, kind="stable")
    return keys[o], ids[o]


@pytest.mark.parametrize("width,height", [(64, 64), (57, 39), (130, 70)])
@pytest.mark.parametrize("n", [1, 2, 33, 127, 129, 511, 513, 640, 1025, 2100])
def test_lists_around_the_round_sizes(n, width, height):
    mean, radius, depth = _items(n, width, height, seed=n)
    keys, ids = _expected(mean, radius, depth, width, height)
    m, r, d = (torch.from_numpy(a).cuda() for a in (mean, radius, depth))
    nt = gs.num_tiles(width, height)
    cap = max(len(ids), 1)
    ws = torch.empty(gs.gs_bin_sort_workspace_size(n, cap, width, height) + 256, device="cuda", dtype=torch.uint8)
    out_k = torch.zeros(cap, device="cuda", dtype=torch.int64)
    out_i = torch.zeros(cap, device="cuda", dtype=torch.int32)
    rng = torch.zeros(2 * nt, device="cuda", dtype=torch.int32)
    _, count = gs.gs_bin_sort(n, m, r, d, width, height, cap, ws, out_k, out_i, rng)
    assert count == len(ids)
    np.testing.assert_array_equal(out_k.cpu().numpy().view(np.uint64)[:count], keys)
    np.testing.assert_array_equal(out_i.cpu().numpy()[:count], ids)
    tiles = (keys >> np.uint64(32)).astype(np.int64)
    per = np.bincount(tiles, minlength=nt)
    got = rng.cpu().numpy().reshape(-1, 2)
    np.testing.assert_array_equal(got[:, 1] - got[:, 0], per)
    # no keys, no synchronisation
    out_i.zero_()
    cnt = torch.zeros(1, device="cuda", dtype=torch.int64)
    gs.gs_bin_sort_views(1, n, m, r, d, [width], [height], cap, ws, None, out_i, rng, count_dev=cnt)
    assert gs.gs_sync_status() == gs.GS_OK and int(cnt) == len(ids)
    np.testing.assert_array_equal(out_i.cpu().numpy()[:count], ids)
    # cut off: the count is reported and nothing is written past the capacity
    if len(ids) > 3:
        small = len(ids) * 2 // 3
        guard = torch.full((cap + 64,), -7, device="cuda", dtype=torch.int32)
        gs.gs_bin_sort_views(1, n, m, r, d, [width], [height], small, ws, None, guard, rng, count_dev=cnt)
        assert gs.gs_sync_status() == gs.GS_ERR_CAPACITY and int(cnt) == len(ids)
        assert (guard[small:] == -7).all()
        assert int(rng.max()) <= small
