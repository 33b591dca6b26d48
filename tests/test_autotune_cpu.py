"""The autotuner times the evaluation whose launches its entries shape: the subset sum, which serves
every call that asks for sum |p_Z| (without it most calls go to the elimination tree)."""
import numpy as np
import pytest

from paper_2010_15595_gb300 import autotune, lib


@pytest.mark.parametrize("precision", [lib.PREC_FP64, lib.PREC_TF])
def test_timed_calls_reach_the_subset_sum(monkeypatch, precision):
    subset = []

    def lhaf(A, stream=None, return_error=False, precision=None):
        subset.append(return_error)
        return (1.0, 0.0) if return_error else 1.0

    def lhaf_batch(mats, precision=None, stream=None, return_abs_sum=False):
        subset.append(return_abs_sum)
        return (np.ones(len(mats)), np.ones(len(mats))) if return_abs_sum else np.ones(len(mats))

    monkeypatch.setattr(lib, "lhaf", lhaf)
    monkeypatch.setattr(lib, "lhaf_batch", lhaf_batch)
    monkeypatch.setattr(lib, "set_batch_tuning", lambda *a, **k: None)
    assert autotune._time_lhaf(np.eye(4, dtype=complex), precision, 2) < 1.0
    autotune.tune_batch(4, precision, candidates=(8,), reps=2, count=4, record=False)
    assert len(subset) == 6 and all(subset)
