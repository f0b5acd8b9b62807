"""The length of a frame's runs when the caller leaves it open (seg = 0): a
power of two near the larger of two runs for every resident CTA of the tile
size's fragment kernel and twice the mean bin, at least 32, at most 256.  The
frame's number of work items equals that of a frame with this length asked for,
whatever the tile size (7 CTAs of it per SM for tiles of 16, as many counted for
8, 1 for 32), and its image too."""
import pytest

from paper_1806_05385_gb300 import scenes as S
from tests.test_deferred_fp64_gpu import _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile,per_sm", [(8, 7), (16, 7), (32, 1)])
@pytest.mark.parametrize("triangles,side,offset", [(1000, 256, 0.5), (20000, 700, 0.3), (60000, 1301, 0.3)])
def test_run_length_follows_the_resident_ctas(pr, tile, per_sm, triangles, side, offset):
    import torch
    sc = S.random_triangles(triangles, 7, offset=offset)
    p0, p1 = S.head_poses(2.0, 0.5)
    view = S.View(W=side, H=side, tan_x=0.5, tan_y=0.5, pose0=p0, pose1=p1, mode=S.MODE_BOTH, fovea=(0.45, 0.55))
    h = pr.pr_scene_upload(_dev(sc.pos), _dev(sc.vel), _dev(sc.col), _dev(sc.tri))
    ws = pr.pr_workspace_create()

    def frame(seg):
        ids = torch.empty(side * side, dtype=torch.int32, device="cuda")
        pr.pr_rasterize_batch(ws, [(h, view, ids, None, None)], pr.make_params("zenon", tile, 0, seg))
        return ids, pr.pr_workspace_stats(ws)

    try:
        frame(32)  # room for runs of 32 (otherwise the items' buffer bounds the cut)
        ids, st = frame(0)
        tiles = ((side + tile - 1) // tile) ** 2
        spread = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
        per = max(st["pairs"] // (2 * spread), 2 * st["pairs"] // max(tiles, spread))
        want = 32
        while want < 256 and 2 * want <= per:
            want *= 2
        ids2, st2 = frame(want)
        assert st["items"] == st2["items"], (want, st["pairs"])
        assert torch.equal(ids, ids2)
    finally:
        pr.pr_workspace_free(ws)
        pr.pr_scene_free(h)
