"""A failed launch between the split of an FP32 product's operands and the
product leaves no marks behind for a later product on the same handle."""
import os
import subprocess
import sys

import pytest

CODE = """
import os, sys
sys.path.insert(0, '.')
import torch, paper_2604_22242_gb300 as fx
g = torch.Generator(device='cuda'); g.manual_seed(1)
def matrix(r, c): return fx.colmajor(r, c, torch.float32).copy_(torch.randn(r, c, generator=g, device='cuda'))
def run(h, x, y, w, fail=False):
    z = fx.colmajor(x.shape[0], y.shape[1], torch.float32)
    for k, t in enumerate((x, y, w, z)): fx.fx_expr_bind(h, k, t.data_ptr(), t.shape[0], t.shape[1], t.stride(1))
    fx.fx_expr_set_launch_shape(h, 256, 4, 1, 0)
    if fail: os.environ['FX_INJECT'] = 'launch_fail'
    try: fx.fx_eval(h, 0)
    except fx.FxError: assert fail
    else: assert not fail
    finally: os.environ.pop('FX_INJECT', None)
    torch.cuda.synchronize()
    return z
big = matrix(1500, 64), matrix(64, 1300), matrix(1500, 1300)
small = matrix(300, 2049), matrix(2049, 257), matrix(300, 257)  # several K ranges per tile
for t in big[:2]: t[3, 5] = 1e-39; t[-1, -1] = 1e-39
used, new = (fx.fx_expr_create('gemm_epilogue', fx.FX_F32) for _ in range(2))
run(used, *big)
run(used, *big, fail=True)
assert torch.equal(run(used, *small), run(new, *small))
print('same')
"""


@pytest.mark.gpu
def test_failed_launch_leaves_no_marks(fxlib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", CODE], cwd=root, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and "same" in out.stdout, out.stdout + out.stderr[-2000:]
