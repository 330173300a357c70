"""Images with more supertiles than splats, whose lists are written by smaller blocks:
splats scattered over the image and, half of them, piled up in one supertile, at
counts around the rounds of 256; against a stable sort in numpy, with and without
keys and cut off at the capacity."""
import numpy as np
import pytest
import torch

from paper_2604_02120_gb300 import gs
from test_gpu_fine_lists import _expected

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height", [(2000, 1500), (24000, 12000)])  # 768 and 70500 supertiles
@pytest.mark.parametrize("n", [1, 33, 255, 257, 513, 700])
def test_more_supertiles_than_splats(n, width, height):
    rng = np.random.default_rng(n)
    mean = rng.uniform([0, 0], [width, height], (n, 2)).astype(np.float32)
    spot = rng.random(n) < 0.8
    mean[spot] = rng.uniform([width - 70, height - 50], [width, height], (spot.sum(), 2))
    radius = rng.integers(0, 60, n).astype(np.int32)
    depth = rng.choice(np.linspace(0.5, 3.0, max(2, n // 3)), n).astype(np.float32)  # with ties
    keys, ids = _expected(mean, radius, depth, width, height)
    m, r, d = (torch.from_numpy(a).cuda() for a in (mean, radius, depth))
    nt, cap = gs.num_tiles(width, height), max(len(ids), 1)
    ws = torch.full((gs.gs_bin_sort_workspace_size(n, cap, width, height) + 256,), 255, device="cuda",
                    dtype=torch.uint8)
    out_k = torch.zeros(cap, device="cuda", dtype=torch.int64)
    out_i = torch.zeros(cap, device="cuda", dtype=torch.int32)
    rng_t = torch.zeros(2 * nt, device="cuda", dtype=torch.int32)
    _, count = gs.gs_bin_sort(n, m, r, d, width, height, cap, ws, out_k, out_i, rng_t)
    assert count == len(ids)
    np.testing.assert_array_equal(out_k.cpu().numpy().view(np.uint64)[:count], keys)
    np.testing.assert_array_equal(out_i.cpu().numpy()[:count], ids)
    got = rng_t.cpu().numpy().reshape(-1, 2)
    np.testing.assert_array_equal(got[:, 1] - got[:, 0],
                                  np.bincount((keys >> np.uint64(32)).astype(np.int64), minlength=nt))
    out_i.zero_()
    cnt = torch.zeros(1, device="cuda", dtype=torch.int64)
    gs.gs_bin_sort_views(1, n, m, r, d, [width], [height], cap, ws, None, out_i, rng_t, count_dev=cnt)
    assert gs.gs_sync_status() == gs.GS_OK and int(cnt) == len(ids)
    np.testing.assert_array_equal(out_i.cpu().numpy()[:count], ids)
    if len(ids) > 3:
        small = len(ids) * 2 // 3
        guard = torch.full((cap + 64,), -7, device="cuda", dtype=torch.int32)
        gs.gs_bin_sort_views(1, n, m, r, d, [width], [height], small, ws, None, guard, rng_t, count_dev=cnt)
        assert gs.gs_sync_status() == gs.GS_ERR_CAPACITY and int(cnt) == len(ids)
        assert (guard[small:] == -7).all()
        assert int(rng_t.max()) <= small
