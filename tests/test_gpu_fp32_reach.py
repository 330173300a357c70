"""The FP32 blends leave out, per 8 x 4 pixels, the list entries that cannot reach
alpha >= 1/255 there.  Every tile lists every splat, so most entries are out of
reach of most blocks: images, T_final and n_contrib against a 64-bit walk of the
whole lists, at list lengths around the groups of 32 and batches of 256."""
import numpy as np
import pytest
import torch

from gpu_common import blend_gpu
from paper_2604_02120_gb300 import gs, scenes
from test_gpu_blend_reach import _splats

pytestmark = pytest.mark.gpu
BG = (0.1, 0.2, 0.3)


def _lists(ids, nt):
    n = ids.size
    return dict(tile_ranges=torch.from_numpy(np.stack([np.arange(nt) * n, np.arange(nt) * n + n], 1)
                                             .astype(np.int32).reshape(-1)).cuda(),
                ids=torch.from_numpy(np.tile(ids.astype(np.int32), nt)).cuda())


def _walk(width, height, mean, conic, opac, rgb):
    """Image, T, n_contrib in 64 bits, which pixels no rounding can flip, and the image's error bound."""
    y, x = np.mgrid[0:height, 0:width] + 0.5
    img, T = np.zeros((3, height, width)), np.ones((height, width))
    last, done = np.zeros((height, width), np.int32), np.zeros((height, width), bool)
    clear, tol = np.ones((height, width), bool), np.full((height, width), 1e-5)
    rel = np.zeros((height, width))  # of T
    for i in range(len(opac)):
        m, k, o, c = (np.asarray(v[i], np.float64) for v in (mean, conic, opac, rgb))
        dx, dy = m[0] - x, m[1] - y
        pw = -0.5 * (k[0] * dx * dx + k[2] * dy * dy) - k[1] * dx * dy
        # FP32 products and sums of Eq. 3 (5 roundings), exp and log2 constants
        eps = 2.0**-21 * (0.5 * (k[0] * dx * dx + k[2] * dy * dy) + abs(k[1] * dx * dy) + 2)
        a = np.minimum(0.99, o * np.exp(np.minimum(pw, 0)))
        clear &= done | (np.abs(np.log(np.maximum(255 * a, 1e-300))) > eps)
        on = ~done & (a >= 1 / 255)
        tt = T * (1 - a)
        rel += np.where(on, 2 * a / (1 - a) * eps + 1e-6, 0)
        clear &= ~on | (np.abs(tt - 1e-4) > rel * 1e-4)
        stop = on & (tt < 1e-4)
        done |= stop
        on &= ~stop
        img += np.where(on, a * T, 0) * c[:, None, None]
        tol += np.where(on, 2 * a * T / (1 - a) * eps, 0)
        T = np.where(on, tt, T)
        last = np.where(on, i + 1, last)
    return img + T * np.asarray(BG)[:, None, None], T, last, clear, tol


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 256, 257, 600])
def test_fp32_lists_of_mostly_unreached_splats(n):
    cam = scenes.look_at_camera((0, 0, -3), (0, 0, 0), 53, 37)
    mean, conic, opac, rgb = _splats(n, cam.width, cam.height, seed=100 + n)
    opac[n // 2] = 2.0  # clamped at 0.99
    proj = {k: torch.from_numpy(v).cuda() for k, v in dict(mean2d=mean, conic=conic, rgb=rgb).items()}
    op = torch.from_numpy(opac).cuda()
    bs = _lists(np.arange(n), cam.num_tiles)
    out = blend_gpu(cam, proj, bs, op, "fp32", bg=BG)
    img, T, last, clear, tol = _walk(cam.width, cam.height, mean, conic, opac, rgb)
    assert clear.mean() > 0.5
    np.testing.assert_array_equal(out["n_contrib"].reshape(last.shape)[clear], last[clear])
    assert (np.abs(out["T_final"].reshape(T.shape) - T) <= tol)[clear].all()
    assert (np.abs(out["image"].reshape(img.shape) - img) <= 3 * tol)[:, clear].all()
    # gradient: nothing for the dead, the same as over the lists without them (up to the order of the sums)
    dead = (opac < 1 / 255) | (mean[:, 0] > 4000)
    live = np.flatnonzero(~dead)
    dL = torch.from_numpy(np.random.default_rng(n).normal(size=(3, cam.height, cam.width)).astype(np.float32)).cuda()
    opts = gs.make_opts("fp32", bg=BG)
    grads = []
    for ids in (np.arange(n), live):
        lists = _lists(ids, cam.num_tiles)
        fwd = {k: torch.from_numpy(v).cuda() for k, v in
               blend_gpu(cam, proj, lists, op, "fp32", bg=BG).items()}
        grads.append(gs.blend_backward(cam.width, cam.height, lists, proj, op, opts, fwd, dL))
        assert gs.gs_sync_status() == gs.GS_OK
    for k in grads[0]:
        a, b = grads[0][k], grads[1][k]
        assert not a[torch.from_numpy(dead).cuda()].any(), k
        assert (a - b).abs().max() <= 1e-3 * b.abs().max(), k


def test_fp32_keeps_a_splat_without_a_position():
    """A NaN exponent counts as 0 (alpha = opacity), as a flat splat's does."""
    cam = scenes.look_at_camera((0, 0, -3), (0, 0, 0), 53, 37)
    outs = []
    for mx, k in ((float("nan"), 1.0), (0.0, 0.0)):
        proj = dict(mean2d=torch.tensor([[mx, 0.0]]).cuda(), conic=torch.tensor([[k, 0.0, k]]).cuda(),
                    rgb=torch.tensor([[0.5, 0.2, 0.9]]).cuda())
        outs.append(blend_gpu(cam, proj, _lists(np.zeros(1), cam.num_tiles), torch.tensor([0.4]).cuda(), "fp32", bg=BG))
    for k in outs[0]:
        np.testing.assert_array_equal(outs[0][k], outs[1][k])
    assert (outs[0]["n_contrib"] == 1).all()
