"""The batch autotuner's cache (no GPU): a result is returned for the library, the candidates and the
trial that it was measured with, and for no other."""
import json

import pytest

from paper_0908_4520_gb300 import autotune, inputs

INST = inputs.batch_instances(8)


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    """tune() with its cache in tmp_path and trials that are counted: the last candidate is the fastest."""
    trials = []

    def trial(sample, precision, threads, smem, warp_cells, chunk):
        trials.append((threads, smem, warp_cells))
        return float(len(trials) % len(autotune.CANDIDATES) or len(autotune.CANDIDATES))

    monkeypatch.setattr(autotune, "_CACHE", str(tmp_path / "cache" / "autotune.json"))
    monkeypatch.setattr(autotune, "_trial", trial)
    return trials


def test_a_result_is_found_again(tuner):
    first = autotune.tune(INST)
    n = len(tuner)
    assert n == len(autotune.CANDIDATES)
    assert (first["threads"], first["smem_bytes"], first["warp_cells"]) == autotune.CANDIDATES[-1]
    again = autotune.tune(INST)
    assert len(tuner) == n and again["warp_cells"] == first["warp_cells"]


@pytest.mark.parametrize("change", ["candidates", "library", "device", "sample", "chunk"])
def test_a_result_of_other_circumstances_is_not(tuner, monkeypatch, change):
    autotune.tune(INST)
    n = len(tuner)
    kw = {}
    if change == "candidates":
        monkeypatch.setattr(autotune, "CANDIDATES", autotune.CANDIDATES[1:])
    elif change == "library":
        monkeypatch.setattr(autotune, "_library_digest", lambda: "other kernels")
    elif change == "device":
        monkeypatch.setattr(autotune, "_device_name", lambda: "another device")
    else:
        kw = {change: 7}
    autotune.tune(INST, **kw)
    assert len(tuner) == n + len(autotune.CANDIDATES)


def test_a_cache_of_the_former_key_is_passed_by(tuner):
    """Files whose keys held the mix alone gave shapes of kernels that are no longer there."""
    import hashlib
    import os

    classes = sorted({(d["quadrature"], d["n_eq"], d["nx"] * d["ny"]) for d in INST})
    key = hashlib.sha256(json.dumps(["threads/smem/warp_cells", "f32", classes]).encode()).hexdigest()[:16]
    os.makedirs(os.path.dirname(autotune._CACHE))
    with open(autotune._CACHE, "w") as fh:
        json.dump({f"f32:{key}": {"threads": 64, "smem_bytes": 0, "warp_cells": 0}}, fh)
    assert autotune.tune(INST)["warp_cells"] == autotune.CANDIDATES[-1][2]
    assert len(tuner) == len(autotune.CANDIDATES)
