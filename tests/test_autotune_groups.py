"""What the autotuner times for a group (no GPU): each distinct launch once."""
import json

from paper_0903_3053_gb300 import autotune, mc
from test_autotune import _Group


def test_group_candidates_are_distinct_launches():
    cands = list(autotune.group_candidates())
    # side by side, sizes do not matter; a cluster of one CTA has nothing to share
    launches = ["members" if s == mc.MC_GROUP_SIDE_BY_SIDE else (C, t, None if C == 1 else s) for C, t, s in cands]
    assert len(set(launches)) == len(launches)
    assert launches[0] == "members"  # preferred where times are equal
    for C in (1, 2, 4, 8, 16):
        assert (C, 256, mc.MC_GROUP_FAIR_SHARE) in cands


def test_entries_of_the_earlier_meaning_are_not_used(monkeypatch, tmp_path):
    """A stored split cost of -1 under the former key was a persistent launch."""
    cache = tmp_path / "autotune.json"
    g = _Group()
    cache.write_text(json.dumps({f"group|fake-device|{autotune._signature(g.batches)}|2":
                                 {"cluster": 16, "threads": 64, "split": -1.0, "ms_per_sweep": 1e-9}}))
    monkeypatch.setattr(autotune, "CACHE", str(cache))
    monkeypatch.setattr(autotune, "_gpu_name", lambda: "fake-device")
    monkeypatch.setattr(autotune, "_time", lambda fn, reps: (fn(), 1.0)[1])
    choice = autotune.tune_group(g, n_sweeps=2, reps=1)
    assert not choice["cached"] and g.cfg == (8, 256, mc.MC_GROUP_SIDE_BY_SIDE)
