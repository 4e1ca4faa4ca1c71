"""The tuner on the GPU: a small domain keeps its resident run."""
import numpy as np
import pytest

from paper_1610_01388_gb300 import autotune, lbm
from paper_1610_01388_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_small_domains_are_tuned_against_the_library_s_choice(tmp_path):
    mask = W.channel_mask(4, 64)
    try:
        best, times = autotune.tune("D2Q9", "IR", "F64", mask.size, cache=str(tmp_path / "c"), mask=mask)
        assert times[best] == min(times.values()) and autotune.UNTUNED in times
        # a run in shared memory against launches of single steps
        assert best == autotune.UNTUNED
        assert not lbm.lbm_tuning_is_set("D2Q9", "IR", "F64", mask.size)
    finally:
        lbm.lbm_tuning_clear()


def test_measured_batch_schedules_are_applied(tmp_path):
    mix = [("D2Q9", W.channel_mask(16, 16), dict(model=m, storage="F32", mu_p=0.1, sigma_y=1e-6, m=1e5,
                                                 g=(1e-6, 0.0, 0.0))) for m in ("IR", "PR")]
    try:
        got = autotune.tune_batch(mix, steps=40, cache=str(tmp_path / "c"))
        assert got["seconds_per_step"] == min(got["tried"].values())
        assert np.isfinite(got["seconds_per_step"])
        assert autotune.load_batch(str(tmp_path / "c")) == 2
    finally:
        lbm.lbm_tuning_clear()
