"""Trees that read every matrix plain and transposed on the skewed tiles
(fx/skew.cuh), and the kernels that the rule of sizes picks on both sides of
its lines, against the oracle."""
import pytest

import synth
from harness import run, specs_for
from test_skew import SHAPE, check, fx  # noqa: F401  (fx is the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f64", "bf16", "f16"])
def test_closed_trees_on_skewed_tiles(fx, storage):
    for k, n in enumerate([1, 7, 57, 63, 65, 129, 257]):
        env = synth.operands(70 + k, specs_for("expr1", n, n), storage, "uniform")
        check("expr1", storage, run(fx, "expr1", storage, env, n, n, shape=SHAPE), env, f" at {n}")


@pytest.mark.parametrize("name,storage,R,C", [
    ("expr1", "f32", 1697, 1697), ("expr1", "f32", 1743, 1743), ("expr1", "bf16", 2047, 2047),
    ("expr1", "bf16", 2051, 2051), ("expr1", "f16", 2053, 2053), ("expr1", "f64", 501, 501),
    ("schur_trans_accu", "bf16", 1025, 1025), ("schur_trans_accu", "f16", 1027, 1027),
    ("schur_trans_accu", "bf16", 1145, 1145), ("schur_exp_trans_sqdiff", "f64", 725, 725),
    ("schur_exp_trans_sqdiff", "f64", 63, 9001), ("schur_trans_accu", "f64", 725, 725)])
def test_both_sides_of_the_lines(fx, name, storage, R, C):
    env = synth.operands(R + C, specs_for(name, R, C), storage, "uniform")
    check(name, storage, run(fx, name, storage, env, R, C), env, f" at {R}x{C}")
