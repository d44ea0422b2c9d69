"""A batch whose items the handle has seen can be evaluated in a stream capture
with any launch shape: changing the shape builds and copies nothing."""
import pytest

pytestmark = pytest.mark.gpu

ROWS, COLS = [64, 33, 200, 1, 500, 0], [64, 70, 65, 9, 130, 4]


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_captured_after_a_change_of_shape(fxlib, storage):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fx = fxlib
    dt, code = {"f32": (torch.float32, fx.FX_F32), "bf16": (torch.bfloat16, fx.FX_BF16)}[storage]
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    n = len(ROWS)
    ops = [[torch.randn(max(r * c, 1), generator=g, device="cuda").to(dt) for _ in range(3)]
           for r, c in zip(ROWS, COLS)]
    z = [torch.zeros(max(r * c, 1), device="cuda", dtype=dt) for r, c in zip(ROWS, COLS)]
    s = torch.zeros(n, device="cuda")
    items = (fx.BatchItem * n)()
    for i, it in enumerate(items):
        for k in range(3):
            it.ptr[k] = ops[i][k].data_ptr()
        it.ptr[3], it.ptr[4] = z[i].data_ptr(), s.data_ptr() + 4 * i
        it.rows, it.cols = ROWS[i], COLS[i]
    h = fx.fx_expr_create("schur_trans_accu", code)
    stream = torch.cuda.Stream()
    try:
        for first in (0, 1):
            fx.fx_expr_set_launch_shape(h, 256, 4, 0, first)
            torch.cuda.synchronize()
            fx.fx_eval_batch(h, items, int(stream.cuda_stream), False)
            torch.cuda.synchronize()
            ref = [t.clone() for t in z]
            for pipeline in (0, 1, 2):
                fx.fx_expr_set_launch_shape(h, 256, 4, 0, pipeline)
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    fx.fx_eval_batch(h, items, int(stream.cuda_stream), False)
                for t in z:
                    t.fill_(float("nan"))
                s.fill_(float("nan"))
                graph.replay()
                torch.cuda.synchronize()
                # element by element the kernels evaluate the same tree
                for i in range(n):
                    k = ROWS[i] * COLS[i]
                    assert torch.equal(z[i][:k], ref[i][:k]), (first, pipeline, i)
                assert bool(torch.isfinite(s).all())
    finally:
        torch.cuda.synchronize()
        fx.fx_expr_destroy(h)
