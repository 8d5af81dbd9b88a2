"""The quotients of R's normalized field: a / b from the correctly rounded 1 / b and one residual
correction (Markstein's theorem), the steps of quotient() in k_pyramid.cu, in exact arithmetic."""
import numpy as np


def _fma(a, b, c):
    # products of two 24-bit significands are exact in 64 bits; so is their sum with c here: the residual
    # a - q b cancels all but the last bits, and the correction's two terms lie within 53 bits
    return np.float32(a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64))


def test_corrected_quotient_is_the_rounded_division():
    rng = np.random.default_rng(5)
    n = 1 << 20
    b = (rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(-40, 40, n)).astype(np.float32)
    a = (rng.uniform(-1.0, 1.0, n) * b).astype(np.float32)          # |component| <= norm
    a[::7] = b[::7]                                                 # rho / sqrt(rho^2) of a flat region
    a[3::11] = 0.0
    r = (1.0 / b.astype(np.float64)).astype(np.float32)
    q = (a * r).astype(np.float32)
    got = _fma(_fma(-q, b, a), r, q)
    np.testing.assert_array_equal(got, a / b)
