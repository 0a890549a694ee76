"""The autotuner's cache: an entry is used again with the sources it was measured with, and not with others."""
import json

import torch

from paper_2010_14132_gb300 import autotune as A


def test_choices_are_kept_per_sources(tmp_path, monkeypatch):
    csrc, cache = tmp_path / "csrc", tmp_path / "cache.json"
    csrc.mkdir()
    (csrc / "a.cu").write_text("one")
    # an entry from before the key named the sources
    cache.write_text(json.dumps({"GPU|64x64x48|mixed": {"y_elems": 16}}))
    calls = []
    monkeypatch.setattr(A, "CSRC", str(csrc))
    monkeypatch.setattr(A, "CACHE", str(cache))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda: "GPU")
    monkeypatch.setattr(A, "autotune", lambda *a: (calls.append(a) or {"y_tile": 8}, []))

    def tuned():
        A._sources.cache_clear()   # as in a new process
        return A.tuned_options(64, 64, 48, 1.0, 1.0, None, None, "mixed")

    assert tuned() == {"y_tile": 8} and len(calls) == 1
    assert tuned() == {"y_tile": 8} and len(calls) == 1
    (csrc / "a.cu").write_text("two")
    assert tuned() == {"y_tile": 8} and len(calls) == 2
    (csrc / "a.cu").write_text("one")
    assert tuned() == {"y_tile": 8} and len(calls) == 2
    A._sources.cache_clear()
