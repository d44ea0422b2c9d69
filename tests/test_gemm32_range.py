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


def product_error(fx, X, Y):
    """Largest error of the product in 2^-24 of |X||Y|: with W = -s X Y the
    sigmoid's argument is s times the error, read back to 2^-25 / 2^18 of it."""
    P = X.astype(np.float64) @ Y.astype(np.float64)
    M = np.abs(X).astype(np.float64) @ np.abs(Y).astype(np.float64)
    s = 2.0 ** np.floor(18 - np.log2(np.median(M)))
    W = (-s * P).astype(np.float32)
    z = evaluate(fx, X, Y, W, s).astype(np.float64)
    return np.max(np.abs(np.log(z / (1 - z)) - (s * P + W)) / (s * M)) * 2 ** 24


@pytest.mark.parametrize("k", [1, 32, 64, 300])
def test_worst_operands_and_one_sign(fx, k):
    """The operands whose left-out plane products are largest (2^-24 of a b),
    and terms of one sign, whose cuts add up: four a block of at most 2 2^-24 of
    its sum each, the small products' twenty 2^-7 of that, and a rounding a
    block."""
    bound = 1 + 4 * 2 + 20 * 2 / 128 + (1 + k // 64)
    worst = np.float32(float.fromhex("0x1.00ff8p+0"))
    assert product_error(fx, np.full((130, k), worst), np.full((k, 129), worst)) <= bound
    rng = np.random.default_rng(8)
    X, Y = (rng.uniform(0.01, 1, d).astype(np.float32) for d in ((200, k), (k, 150)))
    assert product_error(fx, X, Y) <= bound


@pytest.mark.parametrize("e", [-58, -60, -62])
def test_small_operands(fx, e):
    """Products near 2^-120: the parts of the operands are normal, but the
    smallest plane products are not."""
    rng = np.random.default_rng(9)
    X, Y = (np.ldexp(rng.uniform(0.5, 1, d).astype(np.float32), e) for d in ((150, 300), (300, 140)))
    W = np.full((150, 140), -0.25, np.float32)
    s = 2.0 ** (2 * -e - 9)
    if s >= 2.0 ** 127:
        s = 2.0 ** 126
    check(evaluate(fx, X, Y, W, s), X, Y, W, s)
