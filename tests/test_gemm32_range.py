"""FP32 products near and beyond the ends of FP32's range (fx/umma32.cuh):
products that overflow give infinities of the sign they have in FP32, never
NaN, and large finite ones keep FP32's accuracy."""
import numpy as np
import pytest

from test_gemm32 import check, evaluate, fx  # noqa: F401  (fx is the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("v", [3e19, 3e20, 1e25, 1e30, 1e38])
def test_overflowing_products_have_their_sign(fx, v):
    """Rows of one sign each: every product of a row has its sign and every sum
    is beyond FP32, so sigmoid(P + W) is 1 or 0."""
    rng = np.random.default_rng(6)
    X, Y = (rng.uniform(1, 2, d).astype(np.float32) * np.float32(v) for d in ((200, 70), (70, 150)))
    X[::3] *= -1
    W = rng.standard_normal((200, 150)).astype(np.float32)
    ref = np.ones((200, 150), np.float32)
    ref[::3] = 0
    assert np.array_equal(evaluate(fx, X, Y, W, 1.0), ref)


@pytest.mark.parametrize("lo,hi", [(2.0 ** 58, 2.0 ** 60), (2.0 ** 59, 2.0 ** 61)])
def test_below_and_across_the_limit(fx, lo, hi):
    """Magnitudes up to the limit that k_split3 checks, and on both sides of
    it, of one sign and of random signs."""
    rng = np.random.default_rng(7)
    for signs in (False, True):
        X, Y = (np.minimum(rng.uniform(lo, hi, d), hi * (1 - 2.0 ** -24)).astype(np.float32)
                for d in ((150, 100), (100, 140)))
        if signs:
            X *= np.where(rng.random(X.shape) < 0.5, -1, 1).astype(np.float32)
        W = rng.standard_normal((150, 140)).astype(np.float32)
        check(evaluate(fx, X, Y, W, 2.0 ** -125), X, Y, W, 2.0 ** -125)


def test_largest_finite_product(fx):
    """a * b just below FP32's largest value: the BF16 parts of a and b round
    up, and their product alone would be infinite."""
    X = np.full((130, 1), 2.0 ** 64 * (1 - 2.0 ** -24), np.float32)
    Y = np.full((1, 129), 2.0 ** 64 * (1 - 2.0 ** -24), np.float32)
    W = np.zeros((130, 129), np.float32)
    check(evaluate(fx, X, Y, W, 2.0 ** -126), X, Y, W, 2.0 ** -126)
