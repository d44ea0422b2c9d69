"""A launch shape that is set is the one that runs: the vectors per thread
decide how many running sums an FP64 reduction keeps, and so its roundings."""
import pytest

pytestmark = pytest.mark.gpu


def test_fp64_unroll_is_honoured(fxlib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fx = fxlib
    R, C = 61, 173  # one or a few terms per running sum: the order of the sums shows
    differ = {4: 0, 8: 0}
    for seed in range(16):
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        x, y = (torch.randn(C, R, generator=g, device="cuda", dtype=torch.float64).t() for _ in range(2))
        ref = (x - y).square().sum()
        got = {}
        for unroll in (2, 4, 8):
            out = torch.zeros(1, 1, device="cuda", dtype=torch.float64)
            h = fx.fx_expr_create("sqdiff_accu", fx.FX_F64)
            try:
                for k, t in enumerate((x, y, out)):
                    fx.fx_expr_bind(h, k, t.data_ptr(), t.shape[0], t.shape[1], max(t.shape[0], 1))
                fx.fx_expr_set_launch_shape(h, 256, unroll, 1, 0)
                assert fx.fx_expr_launch_shape(h) == (256, unroll, 1, 0)
                fx.fx_eval(h, 0)
                torch.cuda.synchronize()
            finally:
                fx.fx_expr_destroy(h)
            got[unroll] = out.item()
            assert abs(out.item() - ref.item()) <= 1e-13 * ref.item()
        for u in differ:
            differ[u] += got[u] != got[2]
    assert differ[4] > 0 and differ[8] > 0, differ
