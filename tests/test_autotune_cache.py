"""The autotuner's cache file, without a GPU: a choice is replayed for the kernels it was timed among, and only those."""
import json
from types import SimpleNamespace

import pytest

from paper_1402_3545_gb300 import autotune


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    """autotune.tune with the library replaced: what it measured and what it set."""
    calls = SimpleNamespace(measured=0, set=[])
    monkeypatch.setenv("TPMG_TUNE_CACHE", str(tmp_path / "tuning.json"))
    monkeypatch.setattr(autotune.torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(autotune.torch.cuda, "get_device_name", lambda d: "GPU")

    def measure(op, prec, nlevels, reps=5):
        calls.measured += 1
        return [3] * nlevels

    monkeypatch.setattr(autotune.tpmg, "autotune", measure)
    monkeypatch.setattr(autotune.tpmg, "set_variant", lambda op, prec, level, v: calls.set.append((level, v)))
    return calls, tmp_path / "tuning.json"


OP = SimpleNamespace(op=None, nx=64, ny=32, nz=16, L=2)


def test_a_stored_choice_is_replayed(tuner):
    calls, _ = tuner
    assert autotune.tune(OP, 1, True) == [3, 3] and calls.measured == 1
    assert autotune.tune(OP, 1, True) == [3, 3] and calls.measured == 1
    assert calls.set == [(1, 3), (2, 3)]


def test_a_choice_among_earlier_kernels_is_measured_again(tuner, monkeypatch):
    calls, path = tuner
    path.write_text(json.dumps({"GPU|64x32x16|L2|prec1|var1": [0, 0]}))  # as stored before the key named the set
    assert autotune.tune(OP, 1, True) == [3, 3] and calls.measured == 1 and not calls.set
    monkeypatch.setattr(autotune, "VARIANT_SET", autotune.VARIANT_SET + 1)
    assert autotune.tune(OP, 1, True) == [3, 3] and calls.measured == 2 and not calls.set
