"""The tuning cache across versions of the kernels: a record without the
current version (ids of kernels that are gone) is measured again and replaced,
a current one is used as it is."""
import json

import pytest

import paper_2512_16278_gb300 as m


@pytest.mark.parametrize("old", [
    {"gram": 3, "jacobi": 5, "ms": {"g3": 4.6}},
    {"gram": -1, "jacobi": 4, "ms": {}, "version": m.TUNE_VERSION - 1},
])
def test_records_of_other_versions_are_measured_again(tmp_path, monkeypatch, old):
    calls, chosen = [], []
    monkeypatch.setattr(m, "mraid_autotune", lambda plan, d, reps: (calls.append(reps) or (0, 4), {"g0": 1.0}))
    monkeypatch.setattr(m, "mraid_set_variant", lambda plan, v: chosen.append(("gram", v)))
    monkeypatch.setattr(m, "mraid_set_eig_variant", lambda plan, v: chosen.append(("eig", v)))
    cache = tmp_path / "tune.json"
    key = m.tune_key(19, 4096, 1024)
    cache.write_text(json.dumps({key: old, "other": {"gram": 1}}))
    assert m.tune(1, None, 19, 4096, 1024, str(cache)) == (0, 4)
    assert len(calls) == 1 and not chosen
    rec = json.loads(cache.read_text())
    assert rec[key]["gram"] == 0 and rec[key]["version"] == m.TUNE_VERSION and rec["other"] == {"gram": 1}
    assert m.tune(1, None, 19, 4096, 1024, str(cache)) == (0, 4)
    assert len(calls) == 1 and chosen == [("gram", 0), ("eig", 4)]
