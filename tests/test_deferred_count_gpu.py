"""The precision form's FP64 shading launch gets the pixels it is for: those
whose FP32 barycentrics may be off by 2e-5, estimated as 2 x 6e-8 x (the
coordinates' magnitude) x (the sheared triangle's extent) / |det|.  Their number
against the same estimate in FP64 for scenes of small, large and mixed
triangles, up to the pixels within 1e-3 of the line (the FP32 estimate near it
is off by its own 2e-5), and none without the precision form."""
import numpy as np
import pytest

from paper_1806_05385_gb300 import scenes as S
from tests.test_deferred_fp64_gpu import _dev, _scene

pytestmark = pytest.mark.gpu


def _estimate(sc, view, ids):
    """The estimated error over 2e-5 of every covered pixel, in FP64."""
    px = np.flatnonzero(ids >= 0)
    u = np.stack([(px % view.W + 0.5) / view.W, (px // view.W + 0.5) / view.H], 1)
    f = np.float32(view.fovea).astype(np.float64)
    e = u - f
    x = f + e * (np.linalg.norm(e, axis=1, keepdims=True) / np.sqrt(2.0)) ** (view.alpha - 1.0)
    t = x @ np.float32(view.d).astype(np.float64)
    d = (2.0 * x - 1.0) * np.float32([view.tan_x, view.tan_y])
    end = lambda pose, p: p @ np.float64(pose)[:3, :3].T + np.float64(pose)[:3, 3]
    s, m = end(view.pose0, np.float64(sc.pos)), end(view.pose1, np.float64(sc.pos) + np.float64(sc.vel))
    tri = sc.tri[ids[px]]
    c = (1.0 - t)[:, None, None] * s[tri] + t[:, None, None] * m[tri]          # [pixel, vertex, xyz]
    a = c[:, :, :2] - d[:, None, :] * c[:, :, 2:]
    extent = np.abs(a).sum(2).max(1)
    mag = np.abs(c[:, :, 2]).max(1) * (1.0 + np.abs(d).sum(1)) + extent
    det = np.linalg.det(np.stack([a[:, 1] - a[:, 0], a[:, 2] - a[:, 0]], 1))
    return 2.0 * 6e-8 * mag * extent / (2e-5 * np.maximum(np.abs(det), 1e-300))


@pytest.mark.parametrize("kind", ["near", "far", "both"])
def test_pixels_left_to_the_fp64_launch(pr, kind):
    import torch
    sc = _scene(kind)
    h = pr.pr_scene_upload(_dev(sc.pos), _dev(sc.vel), _dev(sc.col), _dev(sc.tri))
    p0, p1 = S.head_poses(2.0, 0.5)
    view = S.View(W=640, H=515, tan_x=0.5, tan_y=0.5, pose0=p0, pose1=p1, mode=S.MODE_BOTH, fovea=(0.45, 0.55))
    ws = pr.pr_workspace_create()
    ids = torch.empty(view.W * view.H, dtype=torch.int32, device="cuda")
    rgb = torch.empty(3 * view.W * view.H, device="cuda")
    try:
        pr.pr_rasterize_batch(ws, [(h, view, ids, None, rgb)], pr.make_params("zenon", 0, 1))
        n = pr.pr_debug_deferred(ws)
        r = _estimate(sc, view, ids.cpu().numpy())
        assert (r > 1.001).sum() <= n <= (r > 0.999).sum(), (n, (r > 1.0).sum(), r.size)
        assert 0 < n < r.size
        pr.pr_rasterize_batch(ws, [(h, view, ids, None, rgb)], pr.make_params("zenon", 0, 0))
        assert pr.pr_debug_deferred(ws) == 0
    finally:
        pr.pr_workspace_free(ws)
        pr.pr_scene_free(h)
