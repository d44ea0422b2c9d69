"""FP32 products with elements outside the planes' range (fx/umma32.cuh): the
tiles they lie in run on FP32 fma (fma_tiles), the others on the planes, in one
launch. Edges of its 64 x 128 pieces and K steps of 16, both tile widths of the
kernel that calls it, several K ranges per tile, strided and misaligned
operands, marks in some tile rows and columns and in all of them."""
import numpy as np
import pytest

from test_gemm32 import check, evaluate, fx  # noqa: F401  (fx is the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (63, 127, 15), (64, 128, 16), (65, 129, 17), (5, 300, 64),
                                   (300, 257, 33), (1000, 700, 200), (300, 257, 2049), (2500, 2300, 49)])
@pytest.mark.parametrize("pad", [0, 3])
def test_sizes(fx, m, n, k, pad):
    rng = np.random.default_rng(m + 7 * n + 31 * k)
    X, Y, W = (rng.standard_normal(d).astype(np.float32) for d in ((m, k), (k, n), (m, n)))
    (X if m > n else Y)[0, 0] = 1e-39  # below the planes' range
    s = 1 / np.sqrt(k)
    check(evaluate(fx, X, Y, W, s, pad), X, Y, W, s)


@pytest.mark.parametrize("m,n,k", [(1000, 700, 512), (2500, 2300, 130)])
@pytest.mark.parametrize("rows,cols", [((0,), ()), ((), (-1,)), ((130, 999), (5, 300, 699)), (None, ()), ((), None)])
def test_marked_rows_and_columns(fx, m, n, k, rows, cols):
    rng = np.random.default_rng(m + n + k)
    X, Y, W = (rng.standard_normal(d).astype(np.float32) for d in ((m, k), (k, n), (m, n)))
    X[list(range(m)) if rows is None else list(rows), 7] = 2.0 ** -120
    Y[9, list(range(n)) if cols is None else list(cols)] = -(2.0 ** -110)
    s = 1 / np.sqrt(k)
    check(evaluate(fx, X, Y, W, s), X, Y, W, s)


def test_marks_are_cleared(fx):
    """A product after one with marked tiles, on the same handle, is the one a
    new handle computes: all on the planes, whose roundings differ from fma's."""
    import torch
    rng = np.random.default_rng(13)
    X, Y, W = (rng.standard_normal(d).astype(np.float32) for d in ((700, 300), (300, 600), (700, 600)))
    bad = X.copy()
    bad[::128, 5] = 1e-39

    def colmajor(a):
        t = fx.colmajor(a.shape[0], a.shape[1], torch.float32)
        return t.copy_(torch.from_numpy(a))

    def run(h, x):
        ts = [colmajor(a) for a in (x, Y, W)] + [fx.colmajor(700, 600, torch.float32)]
        for k, t in enumerate(ts):
            fx.fx_expr_bind(h, k, t.data_ptr(), t.shape[0], t.shape[1], t.stride(1))
        fx.fx_expr_set_scalar(h, 0, 0.05)
        fx.fx_expr_set_launch_shape(h, 256, 4, 1, 0)
        fx.fx_eval(h, 0)
        torch.cuda.synchronize()
        return ts[3].cpu().numpy()

    used, new = (fx.fx_expr_create("gemm_epilogue", fx.FX_F32) for _ in range(2))
    try:
        by_fma = run(used, bad)
        after, ref = run(used, X), run(new, X)
    finally:
        fx.fx_expr_destroy(used)
        fx.fx_expr_destroy(new)
    assert np.array_equal(after, ref) and not np.array_equal(by_fma, ref)


def test_infinity_stays_in_its_row(fx):
    rng = np.random.default_rng(12)
    X, Y = (np.abs(rng.standard_normal(d)).astype(np.float32) + 0.5 for d in ((700, 200), (200, 600)))
    W = np.zeros((700, 600), np.float32)
    X[333, 11] = -np.inf
    Y[3, 444] = np.nan
    got = evaluate(fx, X, Y, W, 1e-3)
    with np.errstate(all="ignore"):
        # row by row: an infinity times a matrix is taken apart by some BLAS libraries
        p = np.stack([(x[:, None] * Y.astype(np.float64)).sum(0) for x in X.astype(np.float64)])
        ref = 1 / (1 + np.exp(-1e-3 * p))
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    ok = ~np.isnan(ref)
    assert np.all(got[333][ok[333]] == 0) and np.max(np.abs(got[ok] - ref[ok])) < 1e-6
