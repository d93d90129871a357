"""The autotuner's cache, with the measurement replaced (no GPU needed)."""
import json

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1402_6081_gb300 as lgfm
from paper_1402_6081_gb300 import autotune

BLOCKS = np.array([[0, 0, 0], [1, 0, 0]], dtype=np.int32)


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    """tune() with made-up times (the defaults are fastest); its measurements and cache file."""
    path, measured = tmp_path / "tune.json", []
    monkeypatch.setenv("LGF_TUNE_CACHE", str(path))
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda d: "GPU")

    def time_options(blocks_list, n_b, levels_list, order, precision, opts, reps=5, warmup=2):
        measured.append(dict(opts))
        return 1.0 + len(opts)

    monkeypatch.setattr(autotune, "time_options", time_options)
    monkeypatch.setattr(autotune, "runs_persistent", lambda *a: False, raising=False)
    return lambda: autotune.tune(BLOCKS, 8, 1, 6, lgfm.LGF_FP32), measured, path


def test_entries_of_other_forms_are_searched_again(tuner):
    tune, measured, path = tuner
    # as written before levels 0 and 1 went by sibling groups: a key without the
    # generation, and a choice that pins the form of then
    old = {"GPU|nb8|p%d|L1|B2|P1" % lgfm.LGF_FP32: {"options": {"interval_kernel": 3}, "ms": 1.0, "all": []}}
    path.write_text(json.dumps(old))
    assert tune() == {} and measured
    n = len(measured)
    assert tune() == {} and len(measured) == n   # from the cache
    assert set(old) < set(json.loads(path.read_text()))   # the file's other entries stay


@pytest.mark.parametrize("persistent,values", [(False, {8}), (True, {-1, 8, 16, 32})])
def test_free_sms_values_that_build_different_schedules(tuner, monkeypatch, persistent, values):
    tune, measured, _ = tuner
    monkeypatch.setattr(autotune, "runs_persistent", lambda *a: persistent, raising=False)
    tune()
    assert {o["free_sms"] for o in measured if "free_sms" in o} == values
