"""FP32 products on BF16 planes (fx/umma32.cuh): tile, K block and split
edges, misaligned operands, in-place results, and operands that cannot be
split (infinities, NaN, subnormal parts, magnitudes that would round up)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fx(fxlib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return fxlib


def colmajor(fx, a, pad=0):
    import torch
    t = torch.full((a.shape[1], a.shape[0] + pad), float("nan"), device="cuda")
    t[:, pad:] = torch.from_numpy(np.ascontiguousarray(a.T)).cuda()
    return t[:, pad:].t()  # ld = rows + pad, base `pad` elements in


def evaluate(fx, X, Y, W, s, pad=0, z_is=None):
    import torch
    ts = [colmajor(fx, a, pad) for a in (X, Y, W)]
    z = ts[z_is] if z_is is not None else fx.colmajor(X.shape[0], Y.shape[1], torch.float32)
    h = fx.fx_expr_create("gemm_epilogue", fx.FX_F32)
    out = []
    try:
        for k, t in enumerate(ts + [z]):
            fx.fx_expr_bind(h, k, t.data_ptr(), t.shape[0], t.shape[1], t.stride(1))
        fx.fx_expr_set_scalar(h, 0, s)
        fx.fx_expr_set_launch_shape(h, 256, 4, 1, 0)  # this kernel at any size
        for _ in range(1 if z_is is not None else 2):
            fx.fx_eval(h, 0)
            torch.cuda.synchronize()
            fx.fx_expr_sync_status(h, 0)
            out.append(z.cpu().numpy().copy())
        assert fx.fx_expr_last_launches(h) == 1
    finally:
        fx.fx_expr_destroy(h)
    assert all(np.array_equal(out[0], o, equal_nan=True) for o in out)
    return out[0]


def logit_bound(X, Y, W, s, K):
    """FP32 bound on the error of the argument s*X*Y + W: the product's terms
    each within 2^-24 and their sums within log-many roundings, taken as the
    plain K + 2 roundings of a dot product over sqrt(K) (random signs) times 8."""
    u = 2.0 ** -24
    mag = np.abs(X.astype(np.float64)) @ np.abs(Y.astype(np.float64)) * abs(s) + np.abs(W)
    return u * (8 * np.sqrt(K) + 8) * mag + 1e-30


def check(got, X, Y, W, s):
    a = s * (X.astype(np.float64) @ Y.astype(np.float64)) + W
    ref = 1 / (1 + np.exp(-a))
    # |sigmoid'| <= 1/4, and the FP32 sigmoid's own few ulps of 1
    tol = logit_bound(X, Y, W, s, X.shape[1]) / 4 + 8 * 2.0 ** -24
    assert np.all(np.abs(got - ref) <= tol), float(np.max(np.abs(got - ref) / tol))


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (5, 300, 64), (129, 127, 65), (128, 128, 63),
                                   (64, 48, 1000), (300, 257, 2049), (1000, 700, 512), (2500, 2300, 190)])
@pytest.mark.parametrize("pad", [0, 3])
def test_sizes(fx, m, n, k, pad):
    rng = np.random.default_rng(m + 7 * n + 31 * k)
    X, Y, W = (rng.standard_normal(d).astype(np.float32) for d in ((m, k), (k, n), (m, n)))
    s = 1 / np.sqrt(k)
    check(evaluate(fx, X, Y, W, s, pad), X, Y, W, s)


def test_in_place(fx):
    rng = np.random.default_rng(3)
    X, Y, W = (rng.standard_normal((200, 200)).astype(np.float32) for _ in range(3))
    for z_is in (0, 1, 2):
        check(evaluate(fx, X, Y, W, 0.07, z_is=z_is), X, Y, W, 0.07)


@pytest.mark.parametrize("scale", [2.0 ** -45, 2.0 ** 45])
def test_scales(fx, scale):
    """Small and large operands against cancelling scalars: the planes' small
    products stay normal down to the limit that k_split3 checks."""
    rng = np.random.default_rng(4)
    X, Y = (rng.standard_normal(d).astype(np.float32) for d in ((150, 333), (333, 140)))
    X, Y = X * np.float32(scale), Y * np.float32(scale)
    W = rng.standard_normal((150, 140)).astype(np.float32)
    s = float(scale ** -2 / 16)
    check(evaluate(fx, X, Y, W, s), X, Y, W, s)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3.4e38, 1e-39, 2.0 ** -101, 2.0 ** 127])
@pytest.mark.parametrize("where", ["X", "Y"])
def test_unsplittable_values(fx, value, where):
    rng = np.random.default_rng(5)
    X, Y = (np.round(rng.standard_normal(d) * 8).astype(np.float32) for d in ((200, 70), (70, 150)))
    W = rng.standard_normal((200, 150)).astype(np.float32)
    (X if where == "X" else Y)[37, 41] = value
    got = evaluate(fx, X, Y, W, 0.01)
    with np.errstate(all="ignore"):
        # small whole numbers: every product and sum of the other terms is exact
        p = np.einsum("ik,kj->ikj", X.astype(np.float64), Y.astype(np.float64)).sum(1)
        a = 0.01 * p + W
        ref = 1 / (1 + np.exp(-a))
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    ok = np.isfinite(ref)
    tol = (np.minimum(np.abs(a), 100.0) * 2.0 ** -22 + 2.0 ** -21)[ok]
    assert np.all(np.abs(got[ok] - ref[ok]) <= tol)
    # the flag is cleared: finite operands afterwards take the planes again
    X, Y = np.ones((200, 70), np.float32), np.ones((70, 150), np.float32)
    check(evaluate(fx, X, Y, W, 0.01), X, Y, W, 0.01)
