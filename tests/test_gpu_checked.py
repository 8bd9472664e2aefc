"""The checked build (libpjds_checked.so, device-side extent checks) on the GPU.

The cases run in a child process that loads the checked library
(tests/checked_cases.py): clean runs of every instrumented mapping must leave
the check word at 0 and match the oracle; indices planted out of range in a
device copy of a matrix must be recorded with their code and skipped.
"""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DIAG, OFFSET, COLUMN, ROW, BLOCK = 1, 2, 3, 4, 5


@pytest.fixture(scope="module")
def res():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1112_5588_gb300 import build
    build.build(checked=True)
    env = dict(os.environ, PJDS_LIBRARY="checked")
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "checked_cases.py")], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_clean_runs_leave_the_check_word_at_zero(res):
    assert len(res["clean"]) >= 4 * 3 * 2 * 12
    bad = [c for c in res["clean"] if c[4] != 0 or not c[5]]
    assert not bad, bad[:10]


def test_planted_column_is_recorded_and_skipped(res):
    n = res["n"]
    for cfg, code, idx in res["planted"]["column"] + res["planted"]["ellr_column"] + res["planted"]["spmm_column"]:
        assert code == COLUMN and idx in (n["n_cols"] + 5, n["n_cols"] + 9), (cfg, code, idx)
    assert res["column_rows_changed"] == 1


def test_planted_perm_entry_is_recorded(res):
    n = res["n"]
    for cfg, code, idx in res["planted"]["perm"]:
        assert (code, idx) == (ROW, n["n_rows"] + 7), cfg


def test_planted_offset_is_recorded(res):
    n = res["n"]
    for cfg, code, idx in res["planted"]["offset"]:
        assert code == OFFSET and idx >= n["n_stored"], (cfg, code, idx)


def test_planted_block_length_is_recorded(res):
    # diagonals past the last one (code 1), or the end sentinel's offset (code 2)
    n = res["n"]
    for cfg, code, idx in res["planted"]["block"]:
        assert (code == DIAG and idx >= n["n_max"] + 1) or (code == OFFSET and idx >= n["n_stored"]), (cfg, code, idx)


@pytest.mark.parametrize("name", ["quad", "paired"])
def test_column_is_recorded_where_rows_share_theirs(res, name):
    # the block product with four and with two rows per thread checks every row's columns
    for cfg, code, idx in res["planted"][name + "_column"]:
        assert (code, idx) == (COLUMN, res[name + "_n_cols"] + 11), (cfg, code, idx)
    assert any(c[0] == name for c in res["clean"])


def test_long_rows_of_a_block_product_are_checked(res):
    n = res["zipf"]
    for cfg, code, idx in res["planted"]["long_column"]:
        assert (code, idx) == (COLUMN, n["n_cols"] + 13), (code, idx)
    for cfg, code, idx in res["planted"]["long_block"]:
        assert (code == DIAG and idx >= n["n_max"] + 1) or (code == OFFSET and idx >= n["n_stored"]), (code, idx)


def test_solves_where_cooperative_launches_are_refused(res):
    # a context that does not hold a launch's CTAs at once (here: a limit of the checked build): the solve in
    # launches of its own, to the same residual (kappa below 5, as in test_gpu_krylov.py)
    assert {tuple(c[:2]) for c in res["refused_cg"]} == {(lo, lim) for lo in ("f64", "f32", "bf16") for lim in (0, 8, -1)}
    for lo, limit, rel, outer in res["refused_cg"]:
        assert rel <= 1e-12 and outer >= 1, (lo, limit, rel)


def test_training_where_cooperative_launches_are_refused(res):
    # the same epochs on fewer CTAs: a gradient is the same terms added in another order (1e-6 of it), which Adam
    # turns into at most lr = 1e-3 a step where a gradient is at its rounding, on the mean far less (12 steps)
    (_, want, w), *others = res["refused_train"]
    assert [c[0] for c in others] == [1, 40]
    for limit, hist, v in others:
        assert hist == pytest.approx(want, rel=2e-3), limit
        assert sum(abs(a - b) for a, b in zip(v, w)) / len(w) <= 2e-5, limit
    assert res["refused_train_error"] == -3  # no launch at all: PJDS_ECUDA
