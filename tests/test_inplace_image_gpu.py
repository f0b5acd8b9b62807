"""A training frame whose image goes into the buffer of its own target or
upstream gradient: every pixel's target or gradient is read before the pixel's
colour is written (background pixels, shaded pixels and, in the precision form,
the pixels shaded in FP64), so loss, gradients and image equal those of a frame
with buffers apart.  Ids and image bit for bit; the loss (a sum of up to 2e5
terms in 256 partial sums) within 1e-5 and the gradients within 1e-4 relative or
1e-5 of the largest, the bounds of the other order-of-addition comparisons."""
import numpy as np
import pytest

from paper_1806_05385_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("fp64", [0, 1])
@pytest.mark.parametrize("kind", ["target_rgb", "grad_rgb"])
@pytest.mark.parametrize("offset", [0.3, 0.004])  # large triangles; small ones, whose pixels are shaded in FP64
@pytest.mark.parametrize("size", [(333, 201), (1600, 1001)])  # blocks and strips of four
def test_image_into_its_target(pr, fp64, kind, offset, size):
    import torch
    sc = S.random_triangles(400, 32, offset=offset)
    h = pr.pr_scene_upload(_dev(sc.pos), _dev(sc.vel), _dev(sc.col), _dev(sc.tri))
    p0, p1 = S.head_poses(2.0, 0.5)
    view = S.View(W=size[0], H=size[1], tan_x=0.5, tan_y=0.5, pose0=p0, pose1=p1, mode=S.MODE_BOTH, fovea=(0.45, 0.55))
    n = view.W * view.H
    given = torch.rand(3 * n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    prm = pr.make_params("zenon", 0, fp64)
    ws = pr.pr_workspace_create()

    def frame(rgb, source):
        g = {k: torch.zeros(3 * sc.V, device="cuda") for k in ("dcol", "dpos", "dvel")}
        loss = torch.zeros(1, device="cuda")
        ids = torch.empty(n, dtype=torch.int32, device="cuda")
        extra = dict(loss=loss) if kind == "target_rgb" else {}
        pr.pr_frame_batch(ws, [(h, view, ids, None, rgb)], [{kind: source, **g, **extra}], prm)
        torch.cuda.synchronize()
        return ids, rgb, loss, g

    try:
        apart = frame(torch.empty(3 * n, device="cuda"), given)  # also grows the bins, so that no frame runs twice
        both = given.clone()
        same = frame(both, both)
        assert torch.equal(apart[0], same[0]) and torch.equal(apart[1], same[1])
        assert int((apart[0] >= 0).sum()) > 100 and int((apart[0] < 0).sum()) > 100
        assert torch.allclose(apart[2], same[2], rtol=1e-5)
        for name, a in apart[3].items():
            assert torch.allclose(a, same[3][name], rtol=1e-4, atol=1e-5 * float(a.abs().max()) + 1e-12), name
    finally:
        pr.pr_workspace_free(ws)
        pr.pr_scene_free(h)
