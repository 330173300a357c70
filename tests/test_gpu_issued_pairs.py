"""gs_blend_opts.issued_pairs of one tile's list: 256 x the list entries up to
the end of every chunk evaluated before the tile's exit, entries that reach no
pixel among them.  A chunk is evaluated after the one `stages` before it has been
composited, so a tile whose pixels all stop in its first chunk evaluates no more
than `stages` chunks, however long its list is."""
import pytest
import torch

from paper_2604_02120_gb300 import gs

pytestmark = pytest.mark.gpu
SHAPES = [(32, 2), (32, 4), (16, 4), (16, 6)]


def _issued(live, opacity, chunk, stages, records, variant="fp16_split"):
    """Issued and evaluated pairs of a 16 x 16 image whose list holds a wide splat where `live` is set
    and one that is far away elsewhere."""
    n = len(live)
    live = torch.tensor(live, device="cuda")
    mean = torch.where(live[:, None], 8.0, 4000.0).expand(n, 2).contiguous()
    conic = torch.tensor([1e-4, 0.0, 1e-4], device="cuda").expand(n, 3).contiguous()
    opac, rgb = torch.full((n,), opacity, device="cuda"), torch.full((n, 3), 0.5, device="cuda")
    ids = torch.arange(n, device="cuda", dtype=torch.int32)
    ranges = torch.tensor([0, n], device="cuda", dtype=torch.int32)
    proj = dict(mean2d=mean, conic=conic, rgb=rgb)
    count = torch.zeros(1, device="cuda", dtype=torch.int64)
    rec = gs.pack_splats(proj, opac) if records else None
    opts = gs.make_opts(variant, chunk=chunk, stages=stages, issued_pairs=count, splat_records=rec)
    out = gs.blend_forward(16, 16, dict(tile_ranges=ranges, ids=ids), proj, opac, opts)
    assert gs.gs_sync_status() == gs.GS_OK
    return int(count), int(out["n_contrib"].sum())


@pytest.mark.parametrize("records", [False, True])
@pytest.mark.parametrize("chunk,stages", SHAPES)
@pytest.mark.parametrize("every", [1, 2, 5])
def test_entries_past_the_exit_are_not_counted(chunk, stages, records, every):
    got, evaluated = _issued([i % every == every - 1 for i in range(3000)], 0.99, chunk, stages, records)
    assert 0 < evaluated <= got <= 256 * stages * chunk * every


@pytest.mark.parametrize("records", [False, True])
@pytest.mark.parametrize("chunk,stages", SHAPES)
@pytest.mark.parametrize("live,tail", [(0, 7), (0, 100), (1, 0), (31, 1), (32, 0), (32, 1), (64, 33), (65, 40),
                                       (96, 500)])
def test_whole_lists_are_counted_whole(chunk, stages, records, live, tail):
    for gap in (0, 40):  # entries out of reach in front and behind, or behind alone
        listed = [False] * gap + [True] * live + [False] * tail
        got, _ = _issued(listed, 0.01, chunk, stages, records)
        assert got == 256 * len(listed)
