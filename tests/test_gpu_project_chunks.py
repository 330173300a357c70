"""gs_project_views runs in chunks of Gaussians: every view's outputs equal
gs_project's of that view alone, bit for bit, at counts around a block (128) and
around the chunks of either size (2048 and 131072 Gaussians)."""
import numpy as np
import pytest
import torch

from paper_2604_02120_gb300 import gs, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degree", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 127, 129, 2047, 2049, 4097, 131071, 131073, 300001])
def test_views_equal_single_projections(n, degree):
    g = torch.Generator(device="cuda").manual_seed(n)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    means, scales, quats = r(n, 3) * 0.5, torch.exp(r(n, 3) * 0.5 - 4), r(n, 4)
    sh = r(n, (degree + 1) ** 2, 3) * 0.3
    cams = scenes.ring_cameras(3, 3.0, [(320, 200), (64, 48), (200, 333)])
    V = len(cams)
    f = lambda *s: torch.full(s, -7.0, device="cuda")  # noqa: E731
    i = lambda *s: torch.full(s, -7, device="cuda", dtype=torch.int32)  # noqa: E731
    out = dict(mean2d=f(V * n + 1, 2), conic=f(V * n + 1, 3), depth=f(V * n + 1), radius=i(V * n + 1),
               rgb=f(V * n + 1, 3), tiles_touched=i(V * n + 1))
    gs.gs_project_views(n, means, scales, quats, sh, degree, [gs.make_camera(c) for c in cams], *out.values())
    assert gs.gs_sync_status() == gs.GS_OK
    for v, cam in enumerate(cams):
        one = gs.project(means, scales, quats, sh, degree, cam)
        for k in out:
            np.testing.assert_array_equal(out[k][v * n:(v + 1) * n].cpu().numpy(), one[k].cpu().numpy(), err_msg=k)
    for k in out:  # nothing past the end
        assert (out[k][V * n:] == -7).all()
