"""The autotuner's cache of batched block sizes (no GPU needed)."""
import json

import pytest

torch = pytest.importorskip("torch")

from paper_2312_06102_gb300 import autotune  # noqa: E402


@pytest.mark.parametrize("ms,threads,want", [
    ({"0": 1.0, "512": 1.2, "1024": 1.3}, 0, 0),
    ({"0": 1.2, "512": 1.3, "1024": 1.0}, 1024, 1024),
    # made before the library chose by the sets: it could only be 512 or 1024
    ({"512": 1.0, "1024": 1.3}, 512, None)])
def test_cached_choice_beside_the_library_rule(tmp_path, monkeypatch, ms, threads, want):
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "a GPU")
    monkeypatch.setattr(autotune, "_CACHE", str(tmp_path / "autotune.json"))
    monkeypatch.setattr(autotune, "_MEM", {"mtime": None, "data": {}})
    entry = {autotune._bkey(1000, 300_000): {"threads": threads, "ms": ms}}
    (tmp_path / "autotune.json").write_text(json.dumps(entry))
    assert autotune.cached_batched(1000, 300_000) == want
    assert autotune.cached_batched(1000, 3_000_000) is None
