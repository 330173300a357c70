"""bin/sort when a look-back gives up.  The kernels are built once more with a
look-back limit of 0, so that a wait for a predecessor that is not there at the
second look ends with the timeout status: then every tile list has to be empty
(ids that were never written are not to be read through) and nothing may be
written past the buffers; a call in which no wait gave up has the usual lists."""
import glob
import os
import subprocess

import pytest
import torch

from paper_2604_02120_gb300 import build, gs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def impatient(tmp_path_factory):
    """libgs.so with only binsort.cu compiled anew."""
    d = tmp_path_factory.mktemp("giveup")
    build.build()
    obj, lib = str(d / "binsort.o"), str(d / "libgs_giveup.so")
    subprocess.check_call([build._nvcc(), *build.NVCC_FLAGS, "-DGS_LOOKBACK_LIMIT_NS=0ull", "-c",
                           os.path.join(build.CSRC, "binsort.cu"), "-o", obj])
    rest = [o for o in sorted(glob.glob(os.path.join(build.BUILD, "*.o"))) if os.path.basename(o) != "binsort.o"]
    subprocess.check_call([build._nvcc(), *build.ARCH, "-shared", "-o", lib, obj, *rest])
    return lib


@pytest.mark.parametrize("width,height", [(1280, 720), (20000, 14000)])  # the latter: more than 2^16 supertiles
@pytest.mark.parametrize("tight", [False, True])
@pytest.mark.parametrize("n", [16_000, 1_300_000])
def test_lists_are_empty_after_a_look_back_gave_up(impatient, monkeypatch, n, tight, width, height):
    gen = torch.Generator(device="cuda").manual_seed(n)
    rand = lambda *s: torch.rand(*s, device="cuda", generator=gen)  # noqa: E731
    mean = (rand(n, 2) * torch.tensor([width, height], device="cuda")).contiguous()
    radius = torch.randint(0, 30, (n,), device="cuda", generator=gen, dtype=torch.int32)
    depth, opac = rand(n) * 9 + 0.1, rand(n)
    k = 9.0 / radius.clamp(min=1).float() ** 2
    conic = torch.stack([k, torch.zeros_like(k), k], 1).contiguous()
    nt = gs.num_tiles(width, height)
    kw = dict(conic=conic, power_min=gs.alpha_power_min(opac)) if tight else {}
    args = (1, n, mean, radius, depth, [width], [height])

    def sort(cap, sync, fill):
        ws = torch.full((gs.gs_bin_sort_workspace_size(n, cap, width, height) + 256,), fill, device="cuda",
                        dtype=torch.uint8)
        ids = torch.full((cap + 4096,), -1, device="cuda", dtype=torch.int32)
        ranges = torch.full((2 * nt + 4096,), -1, device="cuda", dtype=torch.int32)
        cnt = torch.zeros(1, device="cuda", dtype=torch.int64)
        out = gs.gs_bin_sort_views(*args, cap, ws, None, ids, ranges[:2 * nt], check=False,
                                   count_dev=None if sync else cnt, **kw)
        return gs.gs_sync_status(), out, ids, ranges, cnt

    _, (_, need), *_ = sort(16, True, 0)
    status, _, want_ids, want_ranges, _ = sort(need, False, 0)
    assert status == gs.GS_OK
    monkeypatch.setattr(gs, "_lib", None)
    gs.load(impatient)
    gave_up = 0
    for rep in range(8):
        # the workspace's old contents are what holes are read as
        status, _, ids, ranges, cnt = sort(need, rep % 2 == 1, (255, 0, 127, 3)[rep // 2])
        assert (ids[need:] == -1).all() and (ranges[2 * nt:] == -1).all()
        if status == gs.GS_OK:
            assert torch.equal(ids, want_ids) and torch.equal(ranges, want_ranges)
        else:
            gave_up += 1
            assert status == gs.GS_ERR_TIMEOUT
            assert (ranges[:2 * nt] == 0).all()
            if nt > 100_000:
                continue
            proj = dict(mean2d=mean, conic=conic, rgb=torch.ones(n, 3, device="cuda"))
            out = gs.blend_forward(width, height, dict(tile_ranges=ranges[:2 * nt], ids=ids), proj, opac,
                                   gs.make_opts("fp16_split", bg=(0.25, 0.5, 0.75)))
            assert gs.gs_sync_status() == gs.GS_OK
            assert (out["T_final"] == 1).all() and (out["n_contrib"] == 0).all()
    assert gave_up > 0 or n < 1_000_000
