"""What the tensor-core blends drop is dead in the variant's own arithmetic: images,
T_final and n_contrib over whole lists against the same call over lists that keep
only the entries whose exponents (gs_tile_power, which drops nothing) reach alpha >=
1/255 at a pixel, bit for bit, for every operand type, either reference pixel and
splats loaded or gathered from records; the gradients up to the order of the sums."""
import numpy as np
import pytest
import torch

from paper_2604_02120_gb300 import gs, scenes
from test_gpu_blend_reach import _splats

pytestmark = pytest.mark.gpu


def _small_splats(n, width, height, seed):
    """Splats of a pixel or so, densely over the image: the ones a bound in pixels hits hardest."""
    rng = np.random.default_rng(seed)
    mean = rng.uniform([-4, -4], [width + 4, height + 4], (n, 2))
    a, b = 1 / np.exp(rng.uniform(-0.8, 1.2, (2, n))) ** 2
    th = rng.uniform(0, np.pi, n)
    c, s = np.cos(th), np.sin(th)
    conic = np.stack([a * c * c + b * s * s, (a - b) * c * s, a * s * s + b * c * c], 1)
    v = (mean, conic, rng.uniform(0.002, 0.99, n), rng.uniform(0, 1, (n, 3)))
    return [np.ascontiguousarray(x, np.float32) for x in v]


@pytest.mark.parametrize("ref_origin", [0, 1])
@pytest.mark.parametrize("variant", ["fp16", "bf16", "fp16_split", "bf16_split", "fp8_split"])
@pytest.mark.parametrize("kind,n", [("mixed", 33), ("mixed", 1500), ("small", 97), ("small", 2000)])
def test_dropped_entries_are_dead(kind, n, variant, ref_origin):
    cam = scenes.look_at_camera((0, 0, -3), (0, 0, 0), 53, 37)
    W, H, nt = cam.width, cam.height, cam.num_tiles
    make = _splats if kind == "mixed" else _small_splats
    mean, conic, opac, rgb = (torch.from_numpy(v).cuda() for v in make(n, W, H, seed=n))
    proj = dict(mean2d=mean, conic=conic, rgb=rgb)
    ids = torch.arange(n, device="cuda", dtype=torch.int32).repeat(nt)
    r0 = torch.arange(nt, device="cuda", dtype=torch.int32) * n
    ranges = torch.stack([r0, r0 + n], 1).reshape(-1).contiguous()
    kw = dict(bg=(0.1, 0.2, 0.3), ref_origin=ref_origin)
    power = torch.zeros(nt, n, 256, device="cuda")
    gs.gs_tile_power(W, H, ranges, ids, mean, conic, opac, gs.make_opts(variant, **kw),
                     torch.arange(nt, device="cuda", dtype=torch.int32), n, power)
    t, p = torch.arange(nt, device="cuda")[:, None], torch.arange(256, device="cuda")[None]
    inside = ((t % cam.tiles_x) * 16 + p % 16 < W) & ((t // cam.tiles_x) * 16 + p // 16 < H)
    # (the exponents are in base 2, with log2 o; half a unit covers ex2's rounding many times over)
    live = ((power >= -8.5) & inside[:, None]).any(2)
    assert 0 < int(live.sum()) < nt * n or n < 100
    cnt = live.sum(1, dtype=torch.int32)
    end = cnt.cumsum(0, dtype=torch.int32)
    ranges2 = torch.stack([end - cnt, end], 1).reshape(-1).contiguous()
    where = live.nonzero()[:, 1].int().contiguous()
    full = dict(tile_ranges=ranges, ids=ids)
    kept = dict(tile_ranges=ranges2, ids=where if where.numel() else ids[:1].contiguous())
    for extra in (dict(), dict(splat_records=gs.pack_splats(proj, opac))):
        opts = gs.make_opts(variant, **kw, **extra)
        a = gs.blend_forward(W, H, full, proj, opac, opts)
        b = gs.blend_forward(W, H, kept, proj, opac, opts)
        assert gs.gs_sync_status() == gs.GS_OK
        assert torch.equal(a["image"], b["image"]) and torch.equal(a["T_final"], b["T_final"])
        y, x = torch.meshgrid(torch.arange(H, device="cuda"), torch.arange(W, device="cuda"), indexing="ij")
        tile = (y // 16) * cam.tiles_x + x // 16
        nc = b["n_contrib"].long()
        pos = where[(end - cnt)[tile].long() + (nc - 1).clamp(min=0)] + 1 if where.numel() else nc
        assert torch.equal(a["n_contrib"], torch.where(nc > 0, pos, torch.zeros_like(pos)).int())
    dL = torch.randn(3, H, W, device="cuda", generator=torch.Generator(device="cuda").manual_seed(n))
    opts = gs.make_opts(variant, **kw)
    ga = gs.blend_backward(W, H, full, proj, opac, opts, a, dL)
    gb = gs.blend_backward(W, H, kept, proj, opac, opts, b, dL)
    assert gs.gs_sync_status() == gs.GS_OK
    for k in ga:  # (the sums of up to 12 tiles in another order)
        assert (ga[k] - gb[k]).abs().max() <= 1e-4 * gb[k].abs().max(), k
