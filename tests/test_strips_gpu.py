"""Strips of the shading and adjoint kernels: a launch over many pixels gives
each warp a strip of four pixel blocks (32 x 4 pixels), a small launch one
block (8 x 4).  Views of every remainder against the strip's size, in a batch
large enough for strips of four, against the same views in calls of their
own: images bit for bit, losses and gradients up to the order of the float
additions (the tolerance of the other order-of-addition tests)."""
import numpy as np
import pytest

from paper_1806_05385_gb300 import scenes as S

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (7, 3), (8, 4), (9, 5), (31, 4), (32, 8), (33, 7), (64, 13), (65, 33), (127, 2), (100, 96)]


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("source", ["grad", "u8"])
def test_strips_equal_single_blocks(pr, mode, source):
    import torch
    # coarse triangles (whole blocks of one triangle) over fine ones (many per block)
    fine = S.random_triangles(1500, 70 + mode, offset=0.1)
    coarse = S.random_triangles(12, 80 + mode)
    sc = S.Scene(*(np.concatenate([a, b]) for a, b in ((fine.pos, coarse.pos), (fine.vel, coarse.vel),
                                                       (fine.col, coarse.col))),
                 np.concatenate([fine.tri, coarse.tri + fine.V]))
    h = pr.pr_scene_upload(_dev(sc.pos), _dev(sc.vel), _dev(sc.col), _dev(sc.tri))
    p0, p1 = S.head_poses(2.0, 0.5)
    # the last view's 44,000 blocks put the batch over the line to strips of four
    views = [S.View(W=W, H=H, tan_x=0.5, tan_y=0.5, pose0=p0, pose1=p1, mode=mode, fovea=(0.45, 0.55))
             for W, H in SIZES + [(1281, 1101)]]
    rng = np.random.default_rng(7)
    ws, ws1 = pr.pr_workspace_create(), pr.pr_workspace_create()

    def outputs(v):
        n = v.W * v.H
        return (torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, device="cuda"),
                torch.empty(3 * n, device="cuda"))

    def gradients(v, src, loss):
        d = dict(zip(("dcol", "dpos", "dvel"), (torch.zeros(3 * sc.V, device="cuda") for _ in range(3))))
        return dict(grad_rgb=src, **d) if source == "grad" else dict(target_u8=src, loss=loss, **d)

    try:
        srcs = [_dev(rng.normal(size=3 * v.W * v.H).astype(np.float32)) if source == "grad" else
                _dev(rng.integers(0, 256, size=3 * v.W * v.H, dtype=np.uint8)) for v in views]
        outs = [outputs(v) for v in views]
        loss = torch.zeros(len(views), device="cuda")
        grads = [gradients(v, s, loss[k:k + 1]) for k, (v, s) in enumerate(zip(views, srcs))]
        pr.pr_frame_batch(ws, [(h, v, *o) for v, o in zip(views, outs)], grads)
        shown = 0
        for k, (v, s) in enumerate(list(zip(views, srcs))[:len(SIZES)]):
            o = outputs(v)
            one = torch.zeros(1, device="cuda")
            g = gradients(v, s, one)
            pr.pr_frame_batch(ws1, [(h, v, *o)], [g])
            assert all(torch.equal(a, b) for a, b in zip(o, outs[k])), (v.W, v.H)
            shown += int((o[0] >= 0).sum())
            for name in ("dcol", "dpos", "dvel"):
                x, y = grads[k][name], g[name]
                assert torch.allclose(x, y, rtol=1e-4, atol=1e-5 * float(y.abs().max()) + 1e-12), (v.W, v.H, name)
            if source == "u8":
                assert torch.allclose(loss[k:k + 1], one, rtol=1e-5)
        assert shown > 1000
    finally:
        pr.pr_workspace_free(ws)
        pr.pr_workspace_free(ws1)
        pr.pr_scene_free(h)
