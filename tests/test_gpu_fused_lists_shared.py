"""gs_project_bin_small where eight, four, two or one lanes share a splat's rows (by
how many splats a thread would get): lists equal to gs_bin_sort's, with full
rectangles and opacity-aware."""
import numpy as np
import pytest
import torch

from paper_2604_02120_gb300 import gs, scenes
from test_gpu_fused_small import _tile_lists

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tight", [False, True])
@pytest.mark.parametrize("n", [3, 30_400, 30_401, 60_801, 121_601])  # 475 tiles: up to 121600 threads
def test_lists_equal_bin_sort(n, tight):
    cam = scenes.look_at_camera((0, 0, -3), (0, 0, 0), 400, 300)
    rng = np.random.default_rng(n)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()  # noqa: E731
    means, scales = t(rng.uniform(-1, 1, (n, 3))), t(np.exp(rng.normal(-4.6, 0.6, (n, 3))))
    quats, sh, op = t(rng.normal(size=(n, 4))), t(rng.uniform(0, 1, (n, 1, 3))), t(rng.uniform(0.002, 0.9, n))
    pmin = gs.alpha_power_min(op) if tight else None
    proj, bs = gs.project_bin_small(means, scales, quats, sh, 0, cam, max_per_tile=8192, power_min=pmin)
    assert gs.gs_sync_status() == gs.GS_OK
    full = gs.BinSorter("cuda").run(proj["mean2d"], proj["radius"], proj["depth"], cam.width, cam.height)
    if tight:
        cap = max(full["n_instances"], 1)
        ws = torch.empty(gs.gs_bin_sort_workspace_size(n, cap, cam.width, cam.height) + 256, device="cuda",
                         dtype=torch.uint8)
        full = dict(ids=torch.zeros(cap, device="cuda", dtype=torch.int32),
                    tile_ranges=torch.zeros(2 * cam.num_tiles, device="cuda", dtype=torch.int32))
        gs.gs_bin_sort_views(1, n, proj["mean2d"], proj["radius"], proj["depth"], [cam.width], [cam.height], cap, ws,
                             None, full["ids"], full["tile_ranges"], conic=proj["conic"], power_min=pmin)
    assert _tile_lists(bs["tile_ranges"].cpu().numpy(), bs["ids"].cpu().numpy()) == \
        _tile_lists(full["tile_ranges"].cpu().numpy(), full["ids"].cpu().numpy())
