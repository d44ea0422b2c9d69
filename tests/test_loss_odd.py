"""The loss over odd row counts: vectors that run from one column into the
next (k_flat), against the oracle, and on both sides of the size from which
they are taken."""
import pytest

import synth
from harness import oracle_outputs, run, scaled_error, tolerance

pytestmark = pytest.mark.gpu

# below and above 2^18 elements; R = 1, 2, 3 modulo 4 and odd modulo 8, an R
# below one vector (which stays on single elements), one column, n % V = 0..3
SHAPES = [(3, 5), (7, 40000), (5, 60000), (511, 130), (513, 511), (1019, 262), (262147, 1), (2050, 131),
          (1021, 513)]


@pytest.fixture(scope="module")
def fx(fxlib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return fxlib


@pytest.mark.parametrize("storage", ["f32", "f64", "bf16", "f16"])
def test_forward(fx, storage):
    for R, C in SHAPES:
        env = synth.operands(R + C, [("X", R, C), ("W", R, C), ("Y", R, C), ("b", R, 1)], storage, "normal_half")
        got = run(fx, "sigmoid_sqloss", storage, env, R, C)
        (rv, rs), = oracle_outputs("sigmoid_sqloss", env).values()
        err, _, bad, _ = scaled_error(got["s"], rv, rs, "f64" if storage == "f64" else "f32")
        assert bad == 0 and err <= tolerance("sigmoid_sqloss", storage, "s"), (R, C, err)
