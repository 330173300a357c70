"""Opacity-aware bin/sort where the duplication's batches and searches can go
wrong: item counts around a tile of 256, items of so many supertile rows that a
tile takes several batches, rows of hundreds of supertiles, needles whose rows
leave gaps between supertiles, and lists cut off at the capacity; against the
FP64 definition."""
import numpy as np
import pytest
import torch

import oracle
from gpu_common import check_tight_lists
from paper_2604_02120_gb300 import gs

pytestmark = pytest.mark.gpu

SHAPES = {"tall": (40, 2100), "wide": (4100, 72), "gaps": (4100, 72), "square": (333, 290)}


def _items(n, kind, seed):
    width, height = SHAPES[kind]
    rng = np.random.default_rng(seed)
    mean = rng.uniform([-8, -8], [width + 8, height + 8], (n, 2)).astype(np.float32)
    if kind == "wide":  # needles along the rows, a little off
        s1, s2, th = rng.uniform(100, 1500, n), rng.uniform(0.3, 3.0, n), rng.uniform(-0.01, 0.01, n)
    elif kind == "gaps":  # thinner than the pixel centres' spacing: a row's tiles start far from where the last one's end
        s1, s2, th = rng.uniform(300, 1500, n), rng.uniform(0.02, 0.2, n), rng.uniform(-0.01, 0.01, n)
    elif kind == "tall":
        s1, s2, th = rng.uniform(1, 700, n), rng.uniform(0.5, 4.0, n), np.pi / 2 + rng.uniform(-0.02, 0.02, n)
    else:
        s1, s2, th = np.exp(rng.uniform(0, 5, n)), np.exp(rng.uniform(-1, 2, n)), rng.uniform(0, np.pi, n)
    c, s, a, b = np.cos(th), np.sin(th), 1 / s1**2, 1 / s2**2
    conic = np.stack([a * c * c + b * s * s, (a - b) * c * s, a * s * s + b * c * c], 1).astype(np.float32)
    radius = np.ceil(3 * np.maximum(s1, s2)).astype(np.int32)
    radius[rng.random(n) < 0.1] = 0
    opac = rng.uniform(0.001, 0.99, n).astype(np.float32)  # some below 1/255
    depth = rng.choice(np.linspace(0.5, 3.0, max(2, n // 3)), n).astype(np.float32)  # with ties
    return width, height, mean, conic, radius, opac, depth


@pytest.mark.parametrize("kind", list(SHAPES))
@pytest.mark.parametrize("n", [1, 3, 255, 256, 257, 900])
def test_opacity_aware_lists_at_the_batch_edges(n, kind):
    width, height, mean, conic, radius, opac, depth = _items(n, kind, seed=n)
    m, c, r, o, d = (torch.from_numpy(v).cuda() for v in (mean, conic, radius, opac, depth))
    pmin = gs.alpha_power_min(o)
    full = oracle.bin_sort(mean.astype(np.float64), radius, depth, width, height)
    ref = oracle.bin_sort(mean.astype(np.float64), radius, depth, width, height, conic=conic,
                          power_min=pmin.cpu().numpy())
    nt, cap = gs.num_tiles(width, height), max(int(full["n_instances"]), 1)
    ws = torch.empty(gs.gs_bin_sort_workspace_size(n, cap, width, height) + 256, device="cuda", dtype=torch.uint8)
    keys = torch.zeros(cap, device="cuda", dtype=torch.int64)
    ids = torch.zeros(cap, device="cuda", dtype=torch.int32)
    ranges = torch.zeros(2 * nt, device="cuda", dtype=torch.int32)
    kw = dict(conic=c, power_min=pmin)
    _, count = gs.gs_bin_sort_views(1, n, m, r, d, [width], [height], cap, ws, keys, ids, ranges, **kw)
    got = dict(keys=keys[:count].cpu().numpy(), ids=ids[:count].cpu().numpy(), tile_ranges=ranges.cpu().numpy())
    # needles: up to a few pairs per mille lie within rounding of the threshold
    check_tight_lists(got, ref, full, max_amb_frac=0.05)
    assert count == int((got["tile_ranges"][1::2] - got["tile_ranges"][0::2]).sum())
    # cut off: the count is reported and nothing is written past the capacity
    if count > 3:
        small = count * 2 // 3
        cnt = torch.zeros(1, device="cuda", dtype=torch.int64)
        guard = torch.full((cap + 64,), -7, device="cuda", dtype=torch.int32)
        gs.gs_bin_sort_views(1, n, m, r, d, [width], [height], small, ws, None, guard, ranges, count_dev=cnt, **kw)
        assert gs.gs_sync_status() == gs.GS_ERR_CAPACITY and int(cnt) == count
        assert (guard[small:] == -7).all()
        assert int(ranges.max()) <= small
