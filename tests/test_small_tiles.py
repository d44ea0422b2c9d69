"""The register tiles that small matrices take by default, and the TMA
tiles that a given blocks_per_sm asks for, at ragged sizes."""
import pytest

import synth
from harness import oracle_outputs, run, scaled_error, specs_for, tolerance

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fx(fxlib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return fxlib


@pytest.mark.parametrize("bps", [0, 1, 2])
@pytest.mark.parametrize("storage", ["f32", "f64", "bf16", "f16"])
@pytest.mark.parametrize("name", ["schur_exp_trans", "schur_exp_trans_sqdiff", "schur_trans_accu", "expr1"])
def test_ragged_tiles(fx, name, storage, bps):
    for k, (R, C) in enumerate([(8, 8), (64, 64), (72, 56), (136, 8), (8, 136), (264, 200)]):
        if name == "expr1":
            C = R
        env = synth.operands(300 + k, specs_for(name, R, C), storage, "uniform")
        got = run(fx, name, storage, env, R, C, shape=(256, 4, bps, 0))
        for key, (rv, rs) in oracle_outputs(name, env).items():
            st = storage if key == "Z" else ("f64" if storage == "f64" else "f32")
            err, _, bad, _ = scaled_error(got[key], rv, rs, st)
            assert bad == 0 and err <= tolerance(name, storage, key), f"{name}/{storage}/{key} {R}x{C}: {err:.3e}"
