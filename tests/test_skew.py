"""Skewed tiles (fx/skew.cuh): trees with a transposed leaf over matrices
whose columns start at every misalignment, against the oracle, at the edges
of tiles, pieces and shifts."""
import pytest

import synth
from harness import oracle_outputs, run, scaled_error, specs_for, tolerance

pytestmark = pytest.mark.gpu

# one row or column, below one 16-byte piece, tile edges and their neighbours,
# the last rows reached only by the shift (57 + 7 and 61 + 3 fill a tile)
SHAPES = [(1, 1), (1, 70), (3, 2), (5, 67), (57, 65), (58, 64), (61, 63), (63, 7), (65, 130),
          (127, 9), (129, 128), (201, 71), (517, 203)]
SHAPE = (256, 4, 1, 0)  # blocks_per_sm given: these tiles at any size


@pytest.fixture(scope="module")
def fx(fxlib):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return fxlib


def check(name, storage, got, env, label):
    for key, (rv, rs) in oracle_outputs(name, env).items():
        st = storage if key == "Z" else ("f64" if storage == "f64" else "f32")
        err, _, bad, _ = scaled_error(got[key], rv, rs, st)
        assert bad == 0 and err <= tolerance(name, storage, key), f"{name}/{storage}/{key}{label}: {err:.3e}"


@pytest.mark.parametrize("storage", ["f32", "f64", "bf16", "f16"])
@pytest.mark.parametrize("name", ["schur_exp_trans", "schur_exp_trans_sqdiff", "schur_trans_accu", "expr2"])
def test_skewed_tiles(fx, name, storage):
    if name == "expr2" and storage != "f32":
        pytest.skip("compiled for FP32")
    for k, (R, C) in enumerate(SHAPES):
        env = synth.operands(40 + k, specs_for(name, R, C), storage, "uniform")
        check(name, storage, run(fx, name, storage, env, R, C, shape=SHAPE), env, f" at {R}x{C}")


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_residues_and_leading_dimensions(fx, storage):
    name, (R, C) = "schur_exp_trans_sqdiff", (70, 67)
    w = 4 if storage == "f32" else 8
    for pad in (1, 2, w - 1):
        # plain leaves and Z with one residue modulo 16 bytes, D with another
        lds = {s: rows + pad + (w if s == "B" else 0) + (1 if s == "D" else 0)
               for s, rows, _ in specs_for(name, R, C)}
        env = synth.operands(60 + pad, specs_for(name, R, C), storage, "uniform", lds=lds)
        check(name, storage, run(fx, name, storage, env, R, C, ldz=R + pad, shape=SHAPE), env, f" pad {pad}")
        # residues that differ: the general tile kernel
        check(name, storage, run(fx, name, storage, env, R, C, ldz=R + pad + 1, shape=SHAPE), env, f" pad {pad}, Z apart")
