"""The FP64 exp, sqrt and division of fx/dmath.cuh: in ulps on the host
(tests/dmath.cu), and their use on the GPU at arguments that leave the fast
ranges (infinities, NaN, zeros, subnormals, overflow)."""
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_ulps_on_host(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc"
                                    if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "dmath")
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", "-I",
           os.path.join(ROOT, "paper_2604_22242_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
           os.path.join(HERE, "dmath.cu"), "-o", exe]
    p = subprocess.run(cmd, capture_output=True, text=True)
    assert p.returncode == 0, p.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    m = re.match(r"exp (\S+) sqrt (\S+) div (\S+) refused \d+ bad (\d+)", r.stdout)
    assert m, r.stdout
    # a correctly rounded result is within 0.5; the table and the last
    # product add a tenth to exp, the corrections' own rounding 2^-10 to the others
    assert float(m[1]) <= 0.6 and float(m[2]) <= 0.501 and float(m[3]) <= 0.501 and m[4] == "0"


@pytest.mark.gpu
def test_outside_the_fast_ranges(fxlib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fx = fxlib
    inf, nan = np.inf, np.nan
    w = np.array([0.0, -0.0, 5e-324, 1e-310, 2.3e-308, 1e-100, 1.0, 2.0, -3.0, 1e200, 1.7e308, inf, -inf, nan])
    v = np.array([0.0, -0.0, 1e-300, -1e-40, 1.0, -1.0, 699.5, -699.5, 700.5, -700.5, 709.7, -709.9,
                  745.5, -745.5, 1e4, -1e4, inf, -inf, nan])
    W, V = (np.ascontiguousarray(a) for a in np.meshgrid(w, v))
    R, C = W.shape[1], W.shape[0]  # column-major views of the same memory
    X, Y = np.full(W.shape, 0.5), np.full(W.shape, 0.25)
    with np.errstate(all="ignore"):
        ref = X * Y + np.sqrt(np.abs(W)) / (1.0 + np.exp(-V))
    dev = [torch.from_numpy(a).cuda() for a in (X, Y, W, V)]
    z = torch.empty(W.shape, dtype=torch.float64, device="cuda")
    h = fx.fx_expr_create("schur_sqrt_sigmoid", fx.FX_F64)
    try:
        for k, t in enumerate(dev + [z]):
            fx.fx_expr_bind(h, k, t.data_ptr(), R, C, R)
        fx.fx_eval(h, 0)
        torch.cuda.synchronize()
    finally:
        fx.fx_expr_destroy(h)
    got = z.cpu().numpy()
    fin = np.isfinite(ref)
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(got[np.isinf(ref)], ref[np.isinf(ref)])
    # five roundings of at most an ulp (2^-52) each, on positive terms
    assert np.max(np.abs(got[fin] - ref[fin]) / ref[fin]) <= 5 * 2.0 ** -52
