"""16-bit products whose operands TMA cannot address (odd leading
dimensions, bases off 16 bytes), copied to aligned ones first
(umma::k_relayout16), with the remainder in the epilogue."""
import numpy as np
import pytest

import synth
from harness import oracle_outputs, run, scaled_error, tolerance

pytestmark = pytest.mark.gpu
SHAPE = (256, 4, 1, 0)  # blocks_per_sm given: this path at any size


@pytest.fixture(scope="module")
def fx(fxlib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return fxlib


def check(got, env, storage, label):
    (rv, rs), = oracle_outputs("gemm_epilogue", env).values()
    err, _, bad, _ = scaled_error(got["Z"], rv, rs, storage)
    assert bad == 0 and err <= tolerance("gemm_epilogue", storage, "Z"), f"{label}: {err:.3e}"
    assert got["_launches"] == 1


@pytest.mark.parametrize("storage", ["bf16", "f16"])
def test_sizes(fx, storage):
    # one element, pieces of 256 rows and their neighbours, tiles and theirs;
    # X alone, Y alone, and both unaligned
    for k, (R, C, K) in enumerate([(1, 1, 1), (3, 2, 257), (257, 255, 64), (129, 257, 63), (255, 40, 256),
                                   (256, 33, 255), (300, 130, 513)]):
        env = synth.operands(200 + k, [("X", R, K), ("Y", K, C), ("W", R, C)], storage, "normal")
        check(run(fx, "gemm_epilogue", storage, env, R, C, shape=SHAPE), env, storage, f"{R}x{C}, K={K}")


@pytest.mark.parametrize("storage", ["bf16", "f16"])
def test_views(fx, storage):
    R, C, K = 96, 72, 80
    for pad in (1, 3):
        lds = {"X": R + pad, "Y": K + 2 * pad, "W": R + pad}
        env = synth.operands(220 + pad, [("X", R, K), ("Y", K, C), ("W", R, C)], storage, "normal", lds=lds)
        check(run(fx, "gemm_epilogue", storage, env, R, C, ldz=R + pad, offset=pad,
                  shape=SHAPE), env, storage, f"pad {pad}")


def test_in_place(fx):
    import torch
    n, K = 130, 130
    rng = np.random.default_rng(1)
    X, Y, W = (torch.from_numpy(rng.standard_normal((n, n)).astype(np.float32)).bfloat16() for _ in range(3))
    ref = torch.sigmoid(0.1 * (X.double() @ Y.double()) + W.double())
    for z_is in range(3):  # n = 130: both operands unaligned
        ts = []
        for a in (X, Y, W):
            t = fx.colmajor(n, n, torch.bfloat16)
            t.copy_(a)
            ts.append(t)
        h = fx.fx_expr_create("gemm_epilogue", fx.FX_BF16)
        try:
            for k, t in enumerate(ts + [ts[z_is]]):
                fx.fx_expr_bind(h, k, t.data_ptr(), n, n, n)
            fx.fx_expr_set_scalar(h, 0, 0.1)
            fx.fx_expr_set_launch_shape(h, *SHAPE)
            fx.fx_eval(h, 0)
            torch.cuda.synchronize()
        finally:
            fx.fx_expr_destroy(h)
        # FP32 accumulation far below the one rounding to BF16 (2^-9 of at most 1)
        assert float((ts[z_is].double().cpu() - ref).abs().max()) <= 2.0 ** -9 + 1e-4
