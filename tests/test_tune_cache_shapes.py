"""The autotuner's cache keeps a shape by what it is: an entry of a library with other
shapes is not taken for one of this library's, one of the same shape at another
place is found, and files of the older form, with a bare index, are timed anew."""
import json

import paper_2411_18183_gb300.tune as tune
from paper_2411_18183_gb300.tune import TuneCache


def test_entries_follow_the_shape(tmp_path, monkeypatch):
    path = str(tmp_path / "tune.json")
    monkeypatch.setattr(tune, "sig_shapes", lambda: [(24, 2), (16, 2), (32, 1)])
    c = TuneCache(path)
    c.put("a", 0.35, 1)
    c.put("b", 0.5, 0)
    c.put("c", 0.7, 2)
    assert [TuneCache(path).get(k) for k in "abc"] == [(0.35, 1), (0.5, 0), (0.7, 2)]
    monkeypatch.setattr(tune, "sig_shapes", lambda: [(16, 8), (32, 1), (8, 16)])
    assert [TuneCache(path).get(k) for k in "abc"] == [None, None, (0.7, 1)]


def test_index_only_files_are_not_trusted(tmp_path):
    path = str(tmp_path / "tune.json")
    with open(path, "w") as f:
        json.dump({"old": [0.35, 2], "bare": 0.5}, f)
    assert TuneCache(path).get("old") is None and TuneCache(path).get("bare") == (0.5, 0)


def test_without_a_library(tmp_path, monkeypatch):
    def missing():
        raise RuntimeError("not built")
    path = str(tmp_path / "tune.json")
    monkeypatch.setattr(tune, "sig_shapes", missing)
    TuneCache(path).put("a", 0.35, 2)
    assert TuneCache(path).get("a") == (0.35, 2)
    monkeypatch.setattr(tune, "sig_shapes", lambda: [(16, 8), (10, 12), (8, 16)])
    assert TuneCache(path).get("a") is None
