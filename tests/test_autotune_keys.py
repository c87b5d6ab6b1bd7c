"""The autotuner's cache: a configuration is taken from it only when it was
measured on the kernel that would run it.  Timings are stand-ins; no GPU."""
import json
from types import SimpleNamespace

import pytest
import torch

from paper_2608_25376_gb300 import autotune, qpath

HANDLE = SimpleNamespace(info={"C": 92, "n": 92 * 92})


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    """The tuner with stand-in launches: the time of a configuration is its replicas per CTA, 0 taking the longest."""
    runs = []

    def launch(*a, replicas_per_cta=0, **k):
        runs.append(replicas_per_cta)
        return SimpleNamespace(run=lambda stream: None, close=lambda: None)

    def time(fn, reps=2):
        fn()
        return float(runs[-1] or 100)

    monkeypatch.setenv("QPATH_AUTOTUNE_CACHE", str(tmp_path / "autotune.json"))
    monkeypatch.setattr(autotune, "_gpu_key", lambda: "GPU/152sm")
    monkeypatch.setattr(autotune, "_time", time)
    monkeypatch.setattr(torch, "zeros", lambda *a, **k: None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: None)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_properties", lambda d: SimpleNamespace(multi_processor_count=152))
    monkeypatch.setattr(qpath, "schedule", lambda *a: None)
    monkeypatch.setattr(qpath, "qp_anneal_ex", launch)
    monkeypatch.setattr(qpath, "qp_batch_create", launch)
    return SimpleNamespace(runs=runs, path=tmp_path / "autotune.json")


def test_choices_of_the_row_kernels_are_measured_again(tuner):
    tuner.path.write_text(json.dumps({
        "GPU/152sm|rows|C96|R1024": {"replicas_per_cta": 16, "ms": {}},
        "GPU/152sm|batch|F2|Cmax96|Cmed96|R32|stagings0,2": {"replicas_per_cta": 16, "ctas": 152, "flags": 0, "ms": {}},
        f"GPU/152sm|batch|F2|Cmax96|Cmed96|R32|stagings0,{qpath.QP_BATCH_D_SHARED}": {
            "replicas_per_cta": 16, "ctas": 152, "flags": 0, "ms": {}}}))
    assert autotune.tune_single(HANDLE, 1024, 5000) == 1
    assert autotune.tune_batch([HANDLE, HANDLE], 32, 5000)[0] == 2


def test_own_choice_is_kept_and_the_launch_rule_competes(tuner):
    assert autotune.tune_single(HANDLE, 1024, 5000) == 1
    assert 0 in tuner.runs
    n = len(tuner.runs)
    assert autotune.tune_single(HANDLE, 1024, 5000) == 1
    assert len(tuner.runs) == n  # from the cache
