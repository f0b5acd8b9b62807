"""The projected filter at the ends of what it accepts: filter widths far below
a display pixel, colours near the largest float, display pixels on both sides of
the distance at which the window's centre no longer serves as the reference of
the weights, and displays without foveation on both sides of two thirds of the
framebuffer's pixels, up to which the taps come from the image."""
import numpy as np
import pytest

from paper_1806_05385_gb300 import scenes as S
from tests.test_parity_gpu import small_case
from tests.test_unfoveate_gpu import TOL, _covered, _unfoveate_gpu

pytestmark = pytest.mark.gpu


def _case(W=131, H=97):
    _, view = small_case(S.MODE_FOVEATED, W=W, H=H)
    return view, np.random.default_rng(5).uniform(size=(3, H, W)).astype(np.float32)


@pytest.mark.parametrize("sigma", [1e-6, 1e-16, 1e-18, 1e-19, 1e-38])
def test_tiny_sigma_takes_the_nearest_sample(pr, oracle, sigma):
    """Any width far below the sample distances gives the nearest sample.  FP32
    and FP64 may take different ones where two are equally near to about
    1e-4 display pixels: one pixel in a thousand at most."""
    view, img = _case()
    Wd, Hd = 172, 127
    g = _unfoveate_gpu(pr, view, img, Wd, Hd, "projected", sigma)
    assert np.isfinite(g).all()
    o, margin = oracle.unfoveate(view, img, Wd, Hd, "projected", sigma)
    bad = (np.abs(g - o.astype(np.float32)).max(axis=0).reshape(-1) > 0) & _covered(view, Wd, Hd) & (margin >= 1e-3)
    assert bad.mean() < 1e-3
    assert np.array_equal(g, _unfoveate_gpu(pr, view, img, Wd, Hd, "projected", 1e-12))


@pytest.mark.parametrize("sigma", [1e-3, 1e-6, 1e-9, 1e-16])
@pytest.mark.parametrize("case", [(S.MODE_CLASSIC, 640, 480, 320, 240), (S.MODE_CLASSIC, 1000, 600, 500, 900),
                                  (S.MODE_FOVEATED, 64, 64, 32, 32), (S.MODE_FOVEATED, 100, 60, 25, 15)])
def test_equally_near_samples_under_a_narrow_filter(pr, case, sigma):
    """Displays whose pixel centres lie midway between samples: whichever of
    them FP32 calls nearest, the pixel is a mean of colours of its window."""
    mode, W, H, Wd, Hd = case
    p0, p1 = S.head_poses(1.0, 0.0)
    view = S.View(W=W, H=H, tan_x=0.5, tan_y=0.5, pose0=p0, pose1=p1, mode=mode, fovea=(0.5, 0.5))
    img = np.random.default_rng(3).uniform(0.25, 0.75, size=(3, H, W)).astype(np.float32)
    g = _unfoveate_gpu(pr, view, img, Wd, Hd, "projected", sigma)
    assert np.isfinite(g).all() and g.min() >= 0.25 * (1 - 1e-6) and g.max() <= 0.75 * (1 + 1e-6)


def test_colours_near_the_largest_float(pr):
    """Colours of 2^110, display pixels up to 16 in the exponent nearer to
    another sample than to the window's centre: the image is 2^110 times the image of colours in [0, 1].  Both pass through
    exponents (qm - q)(2x - qm - q) k with k = Wd^2 log2(e) / (2 sigma^2) =
    4.5e5, whose second factor is rounded at 2^-24: an error of 2^-23 k |qm - q|
    in an exponent, 3e-4 for samples within 4 sigma, twice (the two images)."""
    view, img = _case()
    Wd, Hd = 3 * view.W, 3 * view.H
    one = _unfoveate_gpu(pr, view, img, Wd, Hd, "projected", 0.5)
    big = _unfoveate_gpu(pr, view, img * np.float32(2.0 ** 110), Wd, Hd, "projected", 0.5)
    assert np.isfinite(big).all()
    cov = _covered(view, Wd, Hd).reshape(Hd, Wd)
    assert np.abs(big * np.float32(2.0 ** -110) - one)[:, cov].max() < 1e-3


def test_both_references_match_the_oracle(pr, oracle):
    """Six display pixels per framebuffer pixel and a narrow filter: centres on
    both sides of exp(-16).  The exponents' error as above with k =
    5e6 and samples of one framebuffer pixel apart (0.015 at the most
    stretched): 1e-2."""
    view, img = _case()
    Wd, Hd = 6 * view.W, 6 * view.H
    g = _unfoveate_gpu(pr, view, img, Wd, Hd, "projected", 0.3)
    o, margin = oracle.unfoveate(view, img, Wd, Hd, "projected", 0.3)
    bad = (np.abs(g - o).max(axis=0).reshape(-1) > 1e-2) & _covered(view, Wd, Hd) & (margin >= 1e-3)
    assert np.isfinite(g).all() and not bad.any()


@pytest.mark.parametrize("mode", [S.MODE_CLASSIC, S.MODE_ROLLING])
@pytest.mark.parametrize("size", [(1, 1, 1, 1), (2, 3, 2, 2), (2, 3, 5, 1), (5, 4, 3, 4), (5, 4, 7, 2), (131, 97, 92, 92),
                                  (131, 97, 92, 93), (257, 33, 16, 8), (64, 300, 200, 64), (300, 64, 64, 201)])
def test_taps_from_image_and_table(pr, oracle, mode, size):
    """Both forms against the oracle with the tolerance of the other display
    tests; a constant image stays constant."""
    W, H, Wd, Hd = size
    _, view = small_case(mode, W=W, H=H)
    img = np.random.default_rng(W + 7 * Hd).uniform(size=(3, H, W)).astype(np.float32)
    for sigma in (0.5, 2.0):
        g = _unfoveate_gpu(pr, view, img, Wd, Hd, "projected", sigma)
        o, margin = oracle.unfoveate(view, img, Wd, Hd, "projected", sigma)
        assert not np.any((np.abs(g - o).max(axis=0).reshape(-1) > TOL) & (margin >= 1e-3))
        flat = _unfoveate_gpu(pr, view, np.full_like(img, 0.375), Wd, Hd, "projected", sigma)
        assert np.abs(flat - 0.375).max() < 1e-6
