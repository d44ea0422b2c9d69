"""The batch autotuner reports only what its choice depends on, and entries
that a cache file holds for other kernels are not applied."""
import json

import pytest

import synth
from test_batch import check, fx, run_batch  # noqa: F401  (fx is the fixture)

pytestmark = pytest.mark.gpu


def test_search_and_stale_entries(fx, tmp_path, monkeypatch):
    cache = tmp_path / "tune.json"
    monkeypatch.setenv("FX_TUNE_CACHE", str(cache))
    rows, cols, ops = synth.batch_operands(12, 48, [("A", False), ("B", False), ("C", True)],
                                           lo=16, hi=300)
    got = []
    zs, ss, _ = run_batch(fx, rows, cols, ops, True, tune="search", shape_out=got)
    check(ops, rows, cols, zs, ss, range(len(rows)))
    b, u, s, p = got[0]
    assert p in (0, 1) and s in (0, 1, 2)
    assert p == 1 or (b, u) == (256, 4)
    (key, value), = json.loads(cache.read_text()).items()
    assert value == f"{b},{u},{s},{p}"
    # an entry written when pipeline 0 was the cp.async kernel
    cache.write_text(json.dumps({key.replace("batch tiles|", "batch|"): "512,8,1,0"}))
    again = []
    zs, ss, _ = run_batch(fx, rows, cols, ops, True, tune="cache", shape_out=again)
    check(ops, rows, cols, zs, ss, range(len(rows)))
    assert again[0] == (256, 4, 0, 0)
