"""A cached pick of the autotuner belongs to the kernels it was measured with."""
from types import SimpleNamespace

import pytest

pytest.importorskip("torch")

from tests.test_autotune_logic import REF, _patch, _sample  # noqa: E402


def test_picks_of_other_kernels_are_not_taken_over(monkeypatch, tmp_path):
    from paper_1708_04329_gb300 import autotune

    cache = tmp_path / "tune.json"
    _, timed = _patch(monkeypatch, lambda ix: 100.0)
    first = autotune.tune_all_bins(REF, 200, 5, 100, _sample(1000), cache=cache)
    n = len(timed)
    monkeypatch.setattr(autotune, "_kernels", lambda: "other kernels", raising=False)
    autotune.tune_all_bins(REF, 200, 5, 100, _sample(1000), cache=cache)
    assert len(timed) == 2 * n  # timed again, for the other kernels
    monkeypatch.undo()
    _patch(monkeypatch, lambda ix: 90.0)
    assert autotune.tune_all_bins(REF, 200, 5, 100, _sample(1000), cache=cache) == first  # still there


def test_unroll_picks_of_other_kernels_are_not_taken_over(monkeypatch, tmp_path):
    import torch

    from paper_1708_04329_gb300 import autotune, grim

    plans = []

    def create(index, cand_unroll=0, **kw):
        plans.append(cand_unroll)
        return SimpleNamespace(stage=lambda **kw: None, close=lambda: None)

    monkeypatch.setattr(grim, "grim_plan_create", create)
    monkeypatch.setattr(autotune, "_time", lambda fn, repeats: 1.0)
    monkeypatch.setattr(autotune, "_device_name", lambda: "fake GPU")
    index = SimpleNamespace(desc=SimpleNamespace(num_bins=1000, q=6))
    sample = dict(reads=torch.zeros(9), lens=torch.zeros(3), cand=torch.zeros(5))
    cache = tmp_path / "tune.json"
    for kernels, tuned in (("a", 4), ("a", 4), ("b", 8)):
        monkeypatch.setattr(autotune, "_kernels", lambda k=kernels: k, raising=False)
        autotune.tune_candidate_unroll(index, sample, 7, cache=cache)
        assert len(plans) == tuned
