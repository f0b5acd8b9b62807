"""Places of the tiles in the bins: a CTA of 256 tiles takes its entries and
each tile-size class's work items with one atomic each.  Batches whose tile
counts lie at the edges of such a CTA, with the classes' borders inside one,
against the same views in calls of their own: images bit for bit, and the
numbers of bin entries and work items the sums of the views' own."""
import numpy as np
import pytest

from paper_1806_05385_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# (width, height, tile): tile counts 1, 255, 256, 257, 16, 3, 512, 4, 60, 1
SHAPES = [(8, 8, 8), (17 * 8, 15 * 8, 8), (16 * 8, 16 * 8, 8), (257 * 8, 5, 8), (64, 64, 16), (33, 9, 16),
          (32 * 16, 16 * 16, 16), (64, 64, 32), (190, 300, 32), (1, 1, 32)]


@pytest.mark.parametrize("seg", [0, 1, 7, 1024])
@pytest.mark.parametrize("fov_bound", ["sector", "recursive"])
def test_mixed_tile_classes_equal_single_views(pr, seg, fov_bound):
    """seg: run length of a work item; fov_bound: the paper's bounds change
    the candidate counts after the bound pass, so their offsets come from a
    scan instead of the bound pass's own atomic."""
    import torch
    sc = S.random_triangles(700, 90, offset=0.25)
    h = pr.pr_scene_upload(_dev(sc.pos), _dev(sc.vel), _dev(sc.col), _dev(sc.tri))
    p0, p1 = S.head_poses(2.0, 0.5)
    views = [(S.View(W=W, H=H, tan_x=0.5, tan_y=0.5, pose0=p0, pose1=p1, mode=k % 4, fovea=(0.45, 0.55)), tile)
             for k, (W, H, tile) in enumerate(SHAPES)]
    prm = pr.make_params("zenon", 0, 0, seg, fov_bound)
    ws, ws1 = pr.pr_workspace_create(), pr.pr_workspace_create()

    def entry(v, tile):
        n = v.W * v.H
        return (h, v, torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, device="cuda"),
                torch.empty(3 * n, device="cuda"), tile)

    try:
        batch = [entry(v, t) for v, t in views]
        pr.pr_rasterize_batch(ws, batch, prm)
        got = pr.pr_workspace_stats(ws)
        # left to the library (0), the run length follows the frame's entries
        want = dict(pairs=0, culled=0, **({"items": 0} if seg else {}))
        for e in batch:
            one = entry(e[1], e[5])
            pr.pr_rasterize_batch(ws1, [one], prm)
            assert all(torch.equal(a, b) for a, b in zip(one[2:5], e[2:5])), (e[1].W, e[1].H)
            for k in want:
                want[k] += pr.pr_workspace_stats(ws1)[k]
        assert {k: got[k] for k in want} == want
        assert want["pairs"] > 1000 and got["items"] > 0
        assert seg != 1 or got["items"] == want["pairs"]
    finally:
        pr.pr_workspace_free(ws)
        pr.pr_workspace_free(ws1)
        pr.pr_scene_free(h)
