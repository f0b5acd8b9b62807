"""(i + 1/2) / n by a product with the correctly rounded 1 / n and two fused
multiply-adds (pixel_centre in csrc/pr_internal.cuh) equals the correctly
rounded quotient: every index of a spread of sizes up to 16384, the fused
operations formed in FP64 (their exact values fit it: 24 + 15 bit products)."""
import numpy as np
import pytest


@pytest.mark.parametrize("first", [1, 2, 3, 5, 7, 11, 13, 16])
def test_centre_is_the_rounded_quotient(first):
    f32, f64 = np.float32, np.float64
    for n in list(range(first, 16385, 101)) + [16383, 16384]:
        a = np.arange(n, dtype=f32) + f32(0.5)
        b, rn = f32(n), f32(1.0) / f32(n)
        q = a * rn
        r = (a.astype(f64) - q.astype(f64) * f64(b)).astype(f32)
        got = (q.astype(f64) + r.astype(f64) * f64(rn)).astype(f32)
        assert np.array_equal(got, a / b), n
