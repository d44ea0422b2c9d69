"""Matrix products written over one of their own operands, with operands that
the tensor-core kernels could read in place: several tiles (a tile's store
must not meet another tile's loads), and enough of them for CTA pairs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fx(fxlib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return fxlib


@pytest.mark.parametrize("name,slots", [("gemm_epilogue", 3), ("gemm_scale", 2)])
@pytest.mark.parametrize("storage", ["bf16", "f16", "f32"])
@pytest.mark.parametrize("n", [136, 520, 1024, 2560])
def test_over_an_operand(fx, name, slots, storage, n):
    import torch
    dt = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}[storage]
    code = {"bf16": fx.FX_BF16, "f16": fx.FX_F16, "f32": fx.FX_F32}[storage]
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    vals = [torch.randn(n, n, generator=g, device="cuda").to(dt) for _ in range(slots)]
    s = 1 / float(np.sqrt(n))
    if name == "gemm_epilogue":
        ref = torch.sigmoid(s * (vals[0].double() @ vals[1].double()) + vals[2].double())
        tol = 2.0 ** -9 + 1e-4 if storage != "f32" else 2e-6  # one rounding to storage of at most 1
    else:
        ref = s * (vals[0].double() @ vals[1].double().t())
        # by way of a temporary: two roundings to storage of values below 8
        tol = {"bf16": 2 * 8 * 2.0 ** -9, "f16": 2 * 8 * 2.0 ** -12, "f32": 2e-5}[storage]
    for z_is in range(slots):
        ts = []
        for v in vals:
            t = fx.colmajor(n, n, dt)
            t.copy_(v)
            ts.append(t)
        h = fx.fx_expr_create(name, code)
        try:
            for k, t in enumerate(ts + [ts[z_is]]):
                fx.fx_expr_bind(h, k, t.data_ptr(), n, n, n)
            fx.fx_expr_set_scalar(h, 0, s)
            fx.fx_eval(h, 0)
            torch.cuda.synchronize()
            fx.fx_expr_sync_status(h, 0)
        finally:
            fx.fx_expr_destroy(h)
        assert float((ts[z_is].double() - ref).abs().max()) <= tol, z_is
