"""The binning count pass at the edges of its tasks (32 to 256 consecutive
candidate pairs of a warp): triangles that span many tasks beside ones with a
single candidate, list lengths around a warp and a task, entries that lose all
candidates (the paper's foveation bounds); and the fragment stage's claims of
several runs at once.  Images are the exact nearest hits whatever the tiles,
bounds and runs, so every setting gives the same bits."""
import numpy as np
import pytest

from paper_1806_05385_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _scene(pr, pos, tri):
    import torch
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a, dtype=t)).cuda()
    pos = np.asarray(pos, np.float32)
    return pr.pr_scene_upload(dev(pos, np.float32), dev(0.02 * pos[:, [1, 2, 0]], np.float32),
                              dev(np.ones_like(pos), np.float32), dev(tri, np.int32))


def _frame(pr, ws, scene, view, tile, prm):
    import torch
    n = view.W * view.H
    out = (torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, device="cuda"),
           torch.empty(3 * n, device="cuda"))
    pr.pr_rasterize_batch(ws, [(scene, view, *out, tile)], prm)
    return out


def _view(W, H, mode):
    p0, p1 = S.head_poses(1.0, 0.3)
    return S.View(W=W, H=H, tan_x=0.6, tan_y=0.6 * H / W, pose0=p0, pose1=p1, mode=mode, fovea=(0.4, 0.6))


@pytest.mark.parametrize("mode", [S.MODE_ROLLING, S.MODE_BOTH])
@pytest.mark.parametrize("n", [0, 1, 30, 31, 32, 255, 256, 1500])
def test_large_and_small_triangles_in_one_list(pr, mode, n):
    import torch
    rng = np.random.default_rng(n + 7 * mode)
    big = np.array([[-9, -9, 12], [9, -9, 13], [0, 14, 12]] * 2, np.float32)
    big[3:] += (0.5, -0.5, 3.0)
    c = rng.uniform((-2, -2, 4), (2, 2, 10), (n, 1, 3))
    small = (c + rng.uniform(-0.05, 0.05, (n, 3, 3))).reshape(-1, 3)
    # the large triangles in the middle of the list
    half = 3 * (n // 2)
    pos = np.concatenate([small[:half], big, small[half:]])
    view = _view(401, 277, mode)
    ws = pr.pr_workspace_create()
    h = _scene(pr, pos, np.arange(len(pos)).reshape(-1, 3))
    try:
        want = _frame(pr, ws, h, view, 32, pr.make_params("quad", 0, 0, 0, "sector"))
        assert (want[0] != -1).float().mean() > 0.5
        for tile in (8, 16, 32):
            for bound, fov in (("zenon", "sector"), ("zenon", "recursive"), ("quad", "simple"), ("trivial", "sector")):
                got = _frame(pr, ws, h, view, tile, pr.make_params(bound, 0, 0, 0, fov))
                assert all(torch.equal(a, b) for a, b in zip(got, want)), (tile, bound, fov)
    finally:
        pr.pr_scene_free(h)
        pr.pr_workspace_free(ws)


@pytest.mark.parametrize("tile,side,views", [(16, 2240, 4), (32, 2400, 2)])
def test_claims_of_several_runs(pr, tile, side, views):
    """seg = 1 makes every run count as long, claimed one by one; with runs
    left to the library these frames' are short and many (enough for claims of
    several with a fragment CTA of every resident warp)."""
    import torch
    rng = np.random.default_rng(tile)
    z = rng.uniform(2, 10, (40_000, 1, 1))
    xy = rng.uniform(-0.6, 0.6, (40_000, 1, 2)) + rng.uniform(-0.01, 0.01, (40_000, 3, 2))
    pos = (np.concatenate([xy, np.ones_like(xy[..., :1])], 2) * z).reshape(-1, 3)
    h = _scene(pr, pos, np.arange(len(pos)).reshape(-1, 3))
    view = _view(side, side - 37, S.MODE_ROLLING)
    n = view.W * view.H
    ws = pr.pr_workspace_create()
    try:
        out = {}
        for seg in (0, 1):
            out[seg] = [(torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, device="cuda"))
                        for _ in range(views)]
            pr.pr_rasterize_batch(ws, [(h, view, *o, None, tile) for o in out[seg]],
                                  pr.make_params("zenon", 0, 0, seg, "sector"))
            if seg == 0:
                ctas = 7 if tile == 16 else 1
                assert pr.pr_workspace_stats(ws)["items"] > 2 * 32 * 152 * ctas
        for got, want in zip(out[0], out[1]):
            assert all(torch.equal(a, b) for a, b in zip(got, want))
    finally:
        pr.pr_scene_free(h)
        pr.pr_workspace_free(ws)
