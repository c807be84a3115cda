"""sq.autotune_step against a fake library: the split mixed step has no warp choice to time, and a choice cached for
other kernels or atoms is not taken."""
import json

import pytest

from paper_2006_03697_gb300 import sq
from workloads import tiny_instance


@pytest.fixture
def fake(monkeypatch):
    calls = []
    state = {"split": True, "counts": [0, 0]}

    def tune(h, n_warps=0, wave_tiles=0, reps=0):
        calls.append((n_warps, wave_tiles, reps))
        if reps > 0:
            state["counts"][0 if state["split"] else 1] += reps
        return 1.0 / (1 + n_warps + (wave_tiles > 0)) if reps > 0 else None

    monkeypatch.setattr(sq, "sq_tune_step", tune)
    monkeypatch.setattr(sq, "sq_step_launch_counts", lambda h: (*state["counts"], 0, 0))
    return calls, state


def test_the_split_step_times_the_wave_sizes_only(fake, tmp_path):
    calls, state = fake
    sq.autotune_step(None, tiny_instance(seed=1), sq.SQ_MIXED, cache=tmp_path / "t.json")
    timed = [c[:2] for c in calls if c[2] > 0]
    assert {w for w, _ in timed} == {0} and len(timed) == len(set(timed)) == 3
    calls.clear()
    state["split"] = False
    _, choice, _ = sq.autotune_step(None, tiny_instance(seed=1), sq.SQ_FP64, cache=tmp_path / "t.json")
    assert len([c for c in calls if c[2] > 0]) == 16 and choice["warps"] == 8


def test_a_choice_for_other_kernels_or_atoms_is_timed_anew(fake, tmp_path, monkeypatch):
    calls, _ = fake
    cache = tmp_path / "t.json"
    inst = tiny_instance(seed=1)
    key, _, times = sq.autotune_step(None, inst, sq.SQ_MIXED, cache=cache)
    assert times is not None and key in json.loads(cache.read_text())
    assert sq.autotune_step(None, inst, sq.SQ_MIXED, cache=cache)[2] is None
    assert sq.autotune_step(None, tiny_instance(seed=1, n_atoms=3), sq.SQ_MIXED, cache=cache)[2] is not None
    monkeypatch.setattr(sq, "_step_sources_id", lambda: "other")
    assert sq.autotune_step(None, inst, sq.SQ_MIXED, cache=cache)[2] is not None
