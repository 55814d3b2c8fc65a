"""Stored tuner results belong to the kernels they were measured on."""
import json

import pytest


@pytest.fixture(scope="module")
def P():
    import paper_2111_11924_gb300 as P

    return P


def test_entries_of_other_kernels_miss(P, tmp_path):
    path = tmp_path / "tune.json"
    key = P.TuneCache.key("GB300", 2048, 2, "crt", 4113)
    res = {"tpi": 4, "form": 0, "window": 5, "ms": 3.1}
    path.write_text(json.dumps({key: dict(res, form=1)}))  # as written before entries named their kernels
    cache = P.TuneCache(str(path))
    assert cache.get(key) is None
    cache.put(key, res)
    assert P.TuneCache(str(path)).get(key) == res
    stored = json.loads(path.read_text())
    assert stored[key]["kernels"] == P.load_library().pmk_kernels_id().decode()
    stored[key]["kernels"] = "0" * 16
    path.write_text(json.dumps(stored))
    assert P.TuneCache(str(path)).get(key) is None


def test_kernels_id_follows_the_sources(P, tmp_path, monkeypatch):
    import shutil

    from paper_2111_11924_gb300 import _native_build as NB

    assert P.load_library().pmk_kernels_id().decode() == NB.kernels_id()
    copy = tmp_path / "csrc"
    shutil.copytree(NB.CSRC, copy)
    monkeypatch.setattr(NB, "CSRC", str(copy))
    before = NB.kernels_id()
    with open(copy / "modexp_core.cuh", "a") as f:
        f.write("// changed\n")
    assert NB.kernels_id() != before != NB.kernels_id(("X=1",))
