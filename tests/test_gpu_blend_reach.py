"""The tensor-core blends drop list entries that reach no pixel of a tile.  Every
tile here lists every splat, so most entries of a list are dead (far away, below
1/255, needles passing by): images, T_final and n_contrib (positions in the whole
list) against the oracle, at list lengths around the groups of 32 and chunks of
16 and 32, for every operand type and pipeline shape."""
import numpy as np
import pytest
import torch

from gpu_common import blend_gpu, compare_to_oracle, oracle_blend_on_gpu_params
from paper_2604_02120_gb300 import gs, scenes

pytestmark = pytest.mark.gpu


def _splats(n, width, height, seed):
    """Splats over and around the image; a third of them cannot reach any pixel."""
    rng = np.random.default_rng(seed)
    mean = rng.uniform([-40, -40], [width + 40, height + 40], (n, 2))
    sig = np.exp(rng.uniform(-0.5, 2.0, (n, 2)))
    sig[rng.random(n) < 0.2, 0] = 60.0  # needles
    th = rng.uniform(0, np.pi, n)
    c, s = np.cos(th), np.sin(th)
    a, b = 1 / sig[:, 0] ** 2, 1 / sig[:, 1] ** 2
    conic = np.stack([a * c * c + b * s * s, (a - b) * c * s, a * s * s + b * c * c], 1)
    opac = rng.uniform(0.02, 0.6, n)
    dead = rng.random(n) < 0.33
    opac[dead & (np.arange(n) % 2 == 0)] = 0.003  # below 1/255 everywhere
    mean[dead & (np.arange(n) % 2 == 1)] += 5000.0
    rgb = rng.uniform(0, 1, (n, 3))
    return [np.ascontiguousarray(v, np.float32) for v in (mean, conic, opac, rgb)]


@pytest.mark.parametrize("n", [1, 15, 17, 31, 32, 33, 64, 65, 97, 300])
@pytest.mark.parametrize("variant,chunk,stages", [("fp16_split", 32, 2), ("bf16_split", 16, 4), ("fp8_split", 32, 4),
                                                  ("fp32_persistent", 16, 6), ("bf16_split", 0, 0)])
def test_lists_of_mostly_dead_splats(n, variant, chunk, stages):
    cam = scenes.look_at_camera((0, 0, -3), (0, 0, 0), 53, 37)
    mean, conic, opac, rgb = _splats(n, cam.width, cam.height, seed=n)
    nt = cam.num_tiles
    ids = np.tile(np.arange(n, dtype=np.int32), nt)
    ranges = np.stack([np.arange(nt) * n, np.arange(nt) * n + n], 1).astype(np.int32).reshape(-1)
    proj_np = dict(mean2d=mean, conic=conic, rgb=rgb)
    bs_np = dict(tile_ranges=ranges, ids=ids)
    proj = {k: torch.from_numpy(v).cuda() for k, v in proj_np.items()}
    bs = {k: torch.from_numpy(v).cuda() for k, v in bs_np.items()}
    bg = (0.1, 0.2, 0.3)
    out = blend_gpu(cam, proj, bs, torch.from_numpy(opac).cuda(), variant, bg=bg, chunk=chunk, stages=stages)
    # the same lists without the splats that are dead everywhere: bit for bit the same image,
    # n_contrib counting the whole list's positions
    live = np.flatnonzero((opac >= 1 / 255) & (mean[:, 0] < 4000))
    m = live.size
    ids2 = np.tile(live.astype(np.int32), nt)
    ranges2 = np.stack([np.arange(nt) * m, np.arange(nt) * m + m], 1).astype(np.int32).reshape(-1)
    bs2 = {k: torch.from_numpy(v).cuda() for k, v in dict(tile_ranges=ranges2, ids=ids2 if m else ids).items()}
    out2 = blend_gpu(cam, proj, bs2, torch.from_numpy(opac).cuda(), variant, bg=bg, chunk=chunk, stages=stages)
    np.testing.assert_array_equal(out["image"], out2["image"])
    np.testing.assert_array_equal(out["T_final"], out2["T_final"])
    pos = np.concatenate([[0], live + 1]).astype(np.int32)
    np.testing.assert_array_equal(out["n_contrib"], pos[out2["n_contrib"]])
    # and against the oracle where its rounding model calls the pixel clear (the splats 5000 px
    # away are ill-conditioned in the model, so that may be few)
    ref = oracle_blend_on_gpu_params(cam, dict(proj_np), dict(tile_ranges=ranges2, ids=ids2 if m else ids), opac,
                                     bg=bg, variant="fp8_split" if variant == "fp8_split" else "split")
    compare_to_oracle(out2, ref, 5e-3 if variant == "fp8_split" else 1e-3, max_amb=1.0)
    if variant != "fp8_split" and variant != "fp32_persistent":
        # the gradient drops the same entries: none of theirs is touched
        dL = torch.ones(3, cam.height, cam.width, device="cuda")
        opts = gs.make_opts(variant, bg=bg)
        fwd = {k: torch.from_numpy(v).cuda() for k, v in out.items()}
        g = gs.blend_backward(cam.width, cam.height, bs, proj, torch.from_numpy(opac).cuda(), opts, fwd, dL)
        assert gs.gs_sync_status() == gs.GS_OK
        dead = torch.from_numpy((opac < 1 / 255) | (mean[:, 0] > 4000)).cuda()
        for k, v in g.items():
            assert torch.isfinite(v).all() and not v[dead].any(), k
