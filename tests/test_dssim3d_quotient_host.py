"""The 3D D-SSIM takes exp's argument d2 / c by the rounded reciprocal of c and one
correction with the exact remainder.  In float32 (the fused steps in float64, which
holds their products exactly) that is the correctly rounded quotient on drawn pairs,
and on pairs around the halfway points, where a wrong bit would show first."""
import numpy as np

f32 = np.float32


def _quotient(d2, c):
    y = f32(1.0) / c
    q = d2 * y
    rest = (d2.astype(np.float64) - q.astype(np.float64) * c.astype(np.float64)).astype(f32)
    return (q.astype(np.float64) + rest.astype(np.float64) * y.astype(np.float64)).astype(f32)


def test_the_corrected_quotient_is_the_division():
    rng = np.random.default_rng(1)
    for _ in range(8):
        n = 500_000
        c = (f32(2) ** rng.integers(-59, 41, n).astype(f32) * rng.uniform(1, 2, n).astype(f32)).astype(f32)
        ratio = np.exp(rng.uniform(-12, 5, n))
        d2 = (c.astype(np.float64) * ratio).astype(f32)
        # around (m + 1/2) ulp: the nearest float32 numerators of such a quotient
        q = rng.uniform(1, 2, n).astype(f32)
        half = q.astype(np.float64) + np.spacing(q).astype(np.float64) / 2
        near = (half * c.astype(np.float64)).astype(f32)
        near = np.where(rng.integers(0, 2, n) == 0, near, np.nextafter(near, f32(0)))
        for num in (d2, near):
            np.testing.assert_array_equal(_quotient(num, c), num / c)
