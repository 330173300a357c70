"""gs_blend_autotune_backward times every built ring depth (2, 3, 4, 6): one untimed
call and `reps` timed ones of each."""
import pytest
import torch

from gpu_common import gpu_pipeline
from paper_2604_02120_gb300 import gs, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reps", [1, 3])
def test_every_built_depth_is_timed(reps):
    dev, cam, proj, bs = gpu_pipeline(scenes.tiny_scene(3, n=200, width=64, height=48))
    opts = gs.make_opts("fp16_split")
    fwd = gs.blend_forward(cam.width, cam.height, bs, proj, dev["opacities"], opts)
    dL = torch.ones(3, cam.height, cam.width, device="cuda")
    grads = gs.blend_backward(cam.width, cam.height, bs, proj, dev["opacities"], opts, fwd, dL)
    before = gs.gs_launch_count()
    ms = gs.gs_blend_autotune_backward([cam.width], [cam.height], 0, bs["tile_ranges"], bs["ids"], proj["mean2d"],
                                       proj["conic"], dev["opacities"], proj["rgb"], opts, fwd["T_final"],
                                       fwd["n_contrib"], dL, grads, reps=reps)
    assert gs.gs_launch_count() - before == 4 * (1 + reps)
    assert ms > 0 and opts.bwd_stages in (2, 3, 4, 6)
