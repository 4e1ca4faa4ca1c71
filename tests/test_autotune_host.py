"""The tuner's choices, with measured times made up: it can keep, and record,
what the library runs without an entry."""
import json

import pytest

from paper_1610_01388_gb300 import autotune, lbm
from paper_1610_01388_gb300 import workloads as W

KEY = ("D2Q9", "IR", "F64")


@pytest.fixture(autouse=True)
def clean(monkeypatch):
    monkeypatch.setattr(autotune, "_gpu_name", lambda: "GPU")
    lbm.lbm_tuning_clear()
    yield
    lbm.lbm_tuning_clear()


def test_unset_takes_an_entry_back():
    assert not lbm.lbm_tuning_is_set(*KEY, 256)
    lbm.lbm_tuning_set(*KEY, 8, 256)
    assert lbm.lbm_tuning_is_set(*KEY, 256) and not lbm.lbm_tuning_is_set(*KEY, 512)
    lbm.lbm_tuning_unset(*KEY, 8)
    assert not lbm.lbm_tuning_is_set(*KEY, 256)
    lbm.lbm_tuning_set_batch(*KEY, 0)
    assert lbm.lbm_tuning_batch_is_set(*KEY) and not lbm.lbm_tuning_batch_is_set("D2Q9", "PR", "F64")
    lbm.lbm_tuning_unset_batch(*KEY)
    assert not lbm.lbm_tuning_batch_is_set(*KEY)
    lib = lbm.library()
    for bad in ((7, 1, 0, 8), (0, 5, 0, 8), (0, 1, 9, 8), (0, 1, 0, 63)):
        assert lib.lbm_tuning_unset(*bad) == lbm.LBM_EINVAL
    for bad in ((7, 1, 0), (0, 5, 0), (0, 1, 9)):
        assert lib.lbm_tuning_unset_batch(*bad) == lbm.LBM_EINVAL


@pytest.mark.parametrize("fastest", [autotune.UNTUNED, (512, 1)])
def test_tune_keeps_and_caches_the_fastest(monkeypatch, tmp_path, fastest):
    cache = str(tmp_path / "cache.json")
    shapes = [c for c in autotune.CANDIDATES if c[1] != 2]
    assert autotune.UNTUNED in shapes
    monkeypatch.setattr(autotune, "measure",
                        lambda *a, **k: {c: 1.0 if c == fastest else 2.0 for c in shapes})
    lbm.lbm_tuning_set(*KEY, 8, 128)
    for load in (False, True):
        if load:
            lbm.lbm_tuning_set(*KEY, 8, 128)
            assert autotune.load(cache) == 1
        else:
            assert autotune.tune(*KEY, 256, cache=cache)[0] == fastest
        assert lbm.lbm_tuning_is_set(*KEY, 256) == (fastest != autotune.UNTUNED)
        assert lbm.lbm_tuning_get(*KEY, 256)[0] == (fastest[0] or 256)


def test_caches_without_the_untuned_choice_are_left_out(tmp_path):
    cache = tmp_path / "cache.json"
    cache.write_text(json.dumps({"GPU": {
        "D2Q9/IR/F64/8": {"block": 128, "cells_per_thread": 1, "seconds_per_step": {"128x1": 1e-6}},
        "batch": {"concurrent": False, "D2Q9/IR/F64/8": {"ctas_per_sm": 0, "threads": 256,
                                                         "cells_per_thread": 1}}}}))
    assert autotune.load(str(cache)) == 0 and autotune.load_batch(str(cache)) == 0
    assert not lbm.lbm_tuning_is_set(*KEY, 256) and not lbm.lbm_tuning_batch_is_set(*KEY)


@pytest.mark.parametrize("fastest", [None, 0, 4])
def test_tune_batch_begins_at_and_can_keep_unset_ctas(monkeypatch, tmp_path, fastest):
    cache = str(tmp_path / "cache.json")
    seen = []

    def measure(mix, steps=160):
        ctas = lbm.lbm_tuning_get_batch(*KEY) if lbm.lbm_tuning_batch_is_set(*KEY) else None
        seen.append((ctas, lbm.lbm_tuning_get_batch_concurrency()))
        return 1.0 if seen[-1] == (fastest, True) else 2.0

    monkeypatch.setattr(autotune, "measure_batch", measure)
    lbm.lbm_tuning_set_batch(*KEY, 2)
    mix = [("D2Q9", W.channel_mask(8, 8), dict(model="IR", storage="F64"))]
    got = autotune.tune_batch(mix, cache=cache)
    assert seen[0] == (None, True)             # what an untuned batch runs
    assert got["ctas_per_sm"] == {"D2Q9/IR/F64": fastest}
    for load in (False, True):
        if load:
            lbm.lbm_tuning_set_batch(*KEY, 2)
            assert autotune.load_batch(cache) == 1
        assert lbm.lbm_tuning_batch_is_set(*KEY) == (fastest is not None)
        assert lbm.lbm_tuning_get_batch(*KEY) == (fastest or 0)
