"""The FP32 blends walk a batch whole where nearly all of its first splats reach a
warp's pixels: lists of wide splats, at lengths around the pairs, groups of 32 and
batches (128, then 256) of that walk, alone and followed by a batch out of reach; against a
64-bit walk, with pixels that stop inside a batch."""
import numpy as np
import pytest
import torch

from gpu_common import blend_gpu
from paper_2604_02120_gb300 import scenes
from test_gpu_fp32_reach import BG, _lists, _walk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opacity", [0.006, 0.4])  # every pixel runs to the end; pixels stop after about 18
@pytest.mark.parametrize("tail", [0, 300])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 127, 128, 129, 255, 257, 383, 384, 385, 600, 641])
def test_dense_batches(n, tail, opacity):
    cam = scenes.look_at_camera((0, 0, -3), (0, 0, 0), 53, 37)
    rng = np.random.default_rng(n)
    f = lambda a: np.ascontiguousarray(a, np.float32)  # noqa: E731
    mean = f(rng.uniform([0, 0], [cam.width, cam.height], (n + tail, 2)))
    mean[n:] += 3000
    s = rng.uniform(60, 200, n + tail)
    conic = f(np.stack([1 / s**2, 0.3 / s**2, 1 / s**2], 1))
    opac, rgb = f(opacity * rng.uniform(0.9, 1.1, n + tail)), f(rng.uniform(0, 1, (n + tail, 3)))
    proj = {k: torch.from_numpy(v).cuda() for k, v in dict(mean2d=mean, conic=conic, rgb=rgb).items()}
    out = blend_gpu(cam, proj, _lists(np.arange(n + tail), cam.num_tiles), torch.from_numpy(opac).cuda(), "fp32", bg=BG)
    img, T, last, clear, tol = _walk(cam.width, cam.height, mean, conic, opac, rgb)
    assert clear.mean() > 0.5
    np.testing.assert_array_equal(out["n_contrib"].reshape(last.shape)[clear], last[clear])
    assert (np.abs(out["T_final"].reshape(T.shape) - T) <= tol)[clear].all()
    assert (np.abs(out["image"].reshape(img.shape) - img) <= 3 * tol)[:, clear].all()
