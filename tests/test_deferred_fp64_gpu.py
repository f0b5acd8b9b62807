"""Pixels that the precision form shades in FP64 are listed by the shading
kernel and shaded by a launch of their own.  Scenes of triangles small
against their distance (nearly every pixel listed), of one far and one near
cluster (some listed) and of near ones (none), two views in a batch, one of
them in another size: the frame's image against pr_shade, which shades them
in place, bit for bit; its loss and gradients against the frame with the
same gradient as an upstream image, up to the order of the float additions."""
import numpy as np
import pytest

from paper_1806_05385_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _scene(kind):
    rng = np.random.default_rng(31)
    near = S.random_triangles(400, 32, offset=0.3)
    far = S.random_triangles(6000, 33, offset=0.004)
    if kind == "near":
        return near
    if kind == "far":
        return far
    return S.Scene(*(np.concatenate([a, b]) for a, b in ((near.pos, far.pos), (near.vel, far.vel),
                                                         (near.col, far.col))),
                   np.concatenate([near.tri, far.tri + near.V]))


@pytest.mark.parametrize("kind", ["near", "far", "both"])
@pytest.mark.parametrize("specular", [0.0, 0.3])
def test_listed_pixels_equal_in_place(pr, kind, specular):
    import torch
    sc = _scene(kind)
    h = pr.pr_scene_upload(_dev(sc.pos), _dev(sc.vel), _dev(sc.col), _dev(sc.tri))
    p0, p1 = S.head_poses(2.0, 0.5)
    views = [S.View(W=W, H=H, tan_x=0.5, tan_y=0.5, pose0=p0, pose1=p1, mode=m, fovea=(0.45, 0.55), k_s=specular,
                    shininess=8.0) for W, H, m in ((640, 515, 3), (333, 201, 1))]
    prm = pr.make_params("zenon", 0, 1)
    ws = pr.pr_workspace_create()
    rng = np.random.default_rng(3)
    try:
        outs = [(torch.empty(v.W * v.H, dtype=torch.int32, device="cuda"), torch.empty(v.W * v.H, device="cuda"),
                 torch.empty(3 * v.W * v.H, device="cuda")) for v in views]
        entries = [(h, v, *o) for v, o in zip(views, outs)]
        loss = torch.zeros(2, device="cuda")

        def zeros():
            return dict(zip(("dcol", "dpos", "dvel"), (torch.zeros(3 * sc.V, device="cuda") for _ in range(3))))

        u8 = [_dev(rng.integers(0, 256, size=3 * v.W * v.H, dtype=np.uint8)) for v in views]
        a = [dict(target_u8=t, loss=loss[k:k + 1], **zeros()) for k, t in enumerate(u8)]
        pr.pr_frame_batch(ws, entries, a, prm)
        for v, o in zip(views, outs):
            ids = torch.empty_like(o[0])
            rgb = torch.empty_like(o[2])
            pr.pr_rasterize(h, v, prm, ids, None)
            pr.pr_shade(h, v, ids, rgb)
            assert torch.equal(ids, o[0]) and torch.equal(rgb, o[2])
        assert sum(int((o[0] >= 0).sum()) for o in outs) > 500
        diff = [o[2] - t.float() * (1.0 / 255.0) for o, t in zip(outs, u8)]
        for k, d in enumerate(diff):
            assert torch.allclose(loss[k].double(), (d.double() ** 2).sum(), rtol=1e-5)
        b = [dict(grad_rgb=2.0 * d, **zeros()) for d in diff]
        pr.pr_frame_batch(ws, entries, b, prm)
        for x, y in zip(a, b):
            for name in ("dcol", "dpos", "dvel"):
                assert torch.allclose(x[name], y[name], rtol=1e-4, atol=1e-5 * float(y[name].abs().max()) + 1e-12)
    finally:
        pr.pr_workspace_free(ws)
        pr.pr_scene_free(h)
