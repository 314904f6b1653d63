"""The stored result of a launch-shape sweep belongs to the code and the
candidates it was measured with (no GPU needed: the sweep itself is replaced by
an exception)."""
import json

import pytest

torch = pytest.importorskip("torch")

import paper_1312_0526_gb300 as hp  # noqa: E402
from paper_1312_0526_gb300 import autotune  # noqa: E402


class Swept(Exception):
    pass


@pytest.fixture
def cache(tmp_path, monkeypatch):
    path = tmp_path / "autotune.json"
    monkeypatch.setattr(autotune, "CACHE", str(path))
    monkeypatch.setattr(autotune, "_device_key", lambda torch: "device")

    def sweep(*args):
        raise Swept
    monkeypatch.setattr(hp, "batched_workspace_size", sweep)
    return path


OFF = torch.arange(5, dtype=torch.int64) * 1000  # four buckets of 1,000 keys
KEYS = torch.zeros(4000, dtype=torch.int64)
CLASS = autotune.workload_key(4, 1000, 1230, False)
SHAPE = {"threads": 128, "ctas_per_sm": 2}


def test_a_result_without_its_code_is_not_taken(cache):
    cache.write_text(json.dumps({"device||" + CLASS: {"tuning": SHAPE}}))
    with pytest.raises(Swept):
        autotune.tune(KEYS, OFF)


def test_a_result_of_other_code_or_candidates_is_not_taken(cache, monkeypatch, tmp_path):
    def key(candidates):
        return "||".join(("device", CLASS, autotune.code_key(candidates)))
    cache.write_text(json.dumps({key(autotune.CANDIDATES[1:]): {"tuning": SHAPE}}))
    with pytest.raises(Swept):
        autotune.tune(KEYS, OFF)
    assert autotune.tune(KEYS, OFF, candidates=autotune.CANDIDATES[1:]) == SHAPE
    cache.write_text(json.dumps({key(autotune.CANDIDATES): {"tuning": SHAPE}}))
    assert autotune.tune(KEYS, OFF) == SHAPE
    other = tmp_path / "batched.cu"
    other.write_text("// another kernel\n")
    monkeypatch.setattr(autotune, "SOURCES", [str(other)])
    autotune._source_digest.cache_clear()
    try:
        with pytest.raises(Swept):
            autotune.tune(KEYS, OFF)
    finally:
        autotune._source_digest.cache_clear()
