"""FP64 division and square root are correctly rounded: on the host
(tests/dround.cu), and on the GPU against the CPU's own."""
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_on_host(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc"
                                    if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "dround")
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", "-I",
           os.path.join(ROOT, "paper_2604_22242_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
           os.path.join(HERE, "dround.cu"), "-o", exe]
    p = subprocess.run(cmd, capture_output=True, text=True)
    assert p.returncode == 0, p.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    m = re.match(r"random (\d+) unsure (\d+) bad 0$", r.stdout.strip())
    assert m, r.stdout
    # the fast paths are left only near powers of two
    assert int(m[2]) < int(m[1]) / 512


@pytest.mark.gpu
def test_on_gpu(fxlib):
    """Z = X % Y + sqrt(abs(W)) / (s0 + exp(-V)) with X = 0 and V large is
    sqrt(abs(W)) / s0: one root and one quotient, each rounded once."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fx = fxlib
    rng = np.random.default_rng(5)
    R, C = 4096, 1024

    def run(w, s0):
        W = torch.from_numpy(w).cuda()
        zero, V = torch.zeros_like(W), torch.full_like(W, 800.0)  # exp(-V) = 0
        z = torch.empty_like(W)
        h = fx.fx_expr_create("schur_sqrt_sigmoid", fx.FX_F64)
        try:
            for k, t in enumerate((zero, zero, W, V, z)):
                fx.fx_expr_bind(h, k, t.data_ptr(), R, C, R)
            fx.fx_expr_set_scalar(h, 0, s0)
            fx.fx_eval(h, 0)
            torch.cuda.synchronize()
        finally:
            fx.fx_expr_destroy(h)
        return z.cpu().numpy()

    a = rng.uniform(1, 4, R * C)
    a[::2] = np.square(rng.uniform(1, 2, R * C // 2)) * (1 + 2.0 ** -52)  # roots near ties among them
    for s0 in (1.0, 3.0, 1.7, 1 - 2.0 ** -53, 1 + 2.0 ** -52):
        assert np.array_equal(run(a, s0), np.sqrt(a) / s0), s0
