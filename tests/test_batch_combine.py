"""The sums of a batch: matrices below, at and above the number of partial sums
up to which a warp adds them (else a block of four warps does), empty ones
among them."""
import pytest

pytestmark = pytest.mark.gpu

# 64 x 64 tiles (32 x 64 in FP64) and 8 partial sums a tile: one tile, 31 to 34
# tiles around the limit, an empty matrix, many tiles
ROWS = [64, 5, 2048, 1984, 2112, 0, 3000, 64, 1, 992, 1024, 1056, 2176, 640, 17]
COLS = [64, 7, 64, 64, 64, 10, 1000, 0, 1, 64, 64, 64, 63, 700, 33]


@pytest.mark.parametrize("storage", ["f32", "f64", "bf16"])
@pytest.mark.parametrize("pipeline", [0, 1, 2])
def test_sums(fxlib, storage, pipeline):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fx = fxlib
    dt, code = {"f32": (torch.float32, fx.FX_F32), "f64": (torch.float64, fx.FX_F64),
                "bf16": (torch.bfloat16, fx.FX_BF16)}[storage]
    sdt = torch.float64 if storage == "f64" else torch.float32
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    n = len(ROWS)
    ops = [[torch.randn(max(r * c, 1), generator=g, device="cuda", dtype=torch.float64).to(dt)
            for _ in range(3)] for r, c in zip(ROWS, COLS)]
    z = [torch.zeros(max(r * c, 1), device="cuda", dtype=dt) for r, c in zip(ROWS, COLS)]
    s = torch.full((n,), float("nan"), device="cuda", dtype=sdt)
    items = (fx.BatchItem * n)()
    for i, it in enumerate(items):
        for k in range(3):
            it.ptr[k] = ops[i][k].data_ptr()
        it.ptr[3], it.ptr[4] = z[i].data_ptr(), s.data_ptr() + i * s.element_size()
        it.rows, it.cols = ROWS[i], COLS[i]
    h = fx.fx_expr_create("schur_trans_accu", code)
    try:
        fx.fx_expr_set_launch_shape(h, 256, 4, 0, pipeline)
        fx.fx_eval_batch(h, items, 0, False)
        torch.cuda.synchronize()
    finally:
        fx.fx_expr_destroy(h)
    # element by element up to four roundings, sums exact far below those
    u = 2.0 ** -53 if storage == "f64" else 2.0 ** -24
    for i, (r, c) in enumerate(zip(ROWS, COLS)):
        a, b, t = (x[:r * c].double() for x in ops[i])
        v = a * b + 0.5 * t.view(r, c).t().reshape(-1)
        mag = (a * b).abs().sum() + (0.5 * t).abs().sum()
        assert abs(float(s[i]) - float(v.sum())) <= 6 * u * float(mag), i
