"""The display kernels at their edges: framebuffers narrower than the 5x5
window or the 3-tap rows, tiles and warps cut by the border, displays of one
row or column, against the FP64 oracle.  Tolerances as in
test_unfoveate_gpu: 2e-5 where the preimage lies in the framebuffer, 1e-3
beyond it, and pixels whose discrete choice lies within 1e-3 texels of its
boundary excused (on grids this small many fall on one)."""
import numpy as np
import pytest

from paper_1806_05385_gb300 import scenes as S
from tests.test_parity_gpu import small_case
from tests.test_unfoveate_gpu import TOL, _covered, _unfoveate_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["mip", "projected"])
@pytest.mark.parametrize("mode", [S.MODE_FOVEATED, S.MODE_ROLLING])
@pytest.mark.parametrize("size", [(2, 3, 5, 7), (4, 5, 9, 7), (5, 4, 7, 11), (6, 64, 17, 61), (65, 3, 67, 1),
                                  (64, 65, 1, 33), (129, 66, 33, 9)])
def test_display_edges(pr, oracle, method, mode, size):
    W, H, Wd, Hd = size
    img = np.random.default_rng(W * 1000 + H).uniform(size=(3, H, W)).astype(np.float32)
    _, view = small_case(mode, W=W, H=H)
    g = _unfoveate_gpu(pr, view, img, Wd, Hd, method, 0.7)
    o, margin = oracle.unfoveate(view, img, Wd, Hd, method, 0.7)
    err = np.abs(g - o).max(axis=0).reshape(-1)
    bad = (err > np.where(_covered(view, Wd, Hd), TOL, 1e-3)) & (margin >= 1e-3)
    assert np.isfinite(g).all()
    assert not bad.any(), (err[bad][:5], np.flatnonzero(bad)[:5])
