"""The reciprocal and the reciprocal root of a pivot in the thread-per-test kernels (no GPU
needed): two Newton steps from the FP32 approximation, whose relative error (at most 2^-22) each
step squares (times 3/2 for the root), so that the result lies within two (three) units in the
last place over the pivots' range.  Emulated with separately rounded FP64 operations (the kernel
fuses the multiply-adds, which only rounds less), from start values off by the
whole of the approximation's error bound."""
import numpy as np


def _range():
    rng = np.random.default_rng(5)
    return np.concatenate([10.0 ** rng.uniform(-12, 12, 200000), rng.uniform(0.5, 2.0, 100000),
                           np.array([1.0000001e-12, 1.0, 2.0, 3.0, 1e12, np.nextafter(1.0, 2.0)])])


def test_reciprocal_within_two_ulps():
    v = _range()
    exact = 1.0 / v
    for off in (-2.0 ** -22, 0.0, 2.0 ** -22):
        x = (exact * (1 + off)).astype(np.float32).astype(np.float64)
        for _ in range(2):
            x = x + x * (1.0 - v * x)
        assert np.max(np.abs(x - exact) / np.spacing(exact)) <= 2.0


def test_reciprocal_root_within_three_ulps():
    v = _range()
    exact = 1.0 / np.sqrt(v.astype(np.longdouble))
    for off in (-2.0 ** -22, 0.0, 2.0 ** -22):
        y = (exact * (1 + off)).astype(np.float32).astype(np.float64)
        for _ in range(2):
            y = y + (0.5 * y) * (1.0 - (v * y) * y)
        assert np.max(np.abs(y - exact) / np.spacing(exact.astype(np.float64))) <= 3.0
