"""The autotuner's cache: a decision made for other kernels is not applied."""
import json

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture
def tuner(monkeypatch):
    from paper_2606_04801_gb300 import autotune

    applied, tuned = [], []
    monkeypatch.setattr(autotune, "survivor_fraction", lambda inputs: 0.25)
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda dev: "a GPU")
    monkeypatch.setattr(autotune, "apply", applied.append)

    def tune(inputs):
        tuned.append(1)
        return {"zchunk3d": 64, "ctas3d": 0, "rows2d": 64, "uf_variant": 0}

    monkeypatch.setattr(autotune, "tune", tune)
    return autotune, applied, tuned


def test_a_decision_for_other_kernels_is_made_again(tuner, tmp_path, monkeypatch):
    autotune, applied, tuned = tuner
    vol = [torch.zeros(8, 8, 8)]
    path = tmp_path / "t.json"
    # as written by a library whose keys held no sources, and by one of other sources
    old = f"a GPU|{autotune.bucket([(8, 8, 8)])}|surv:-2"
    stale = {"zchunk3d": 16, "ctas3d": 3, "rows2d": 64, "uf_variant": 1}
    path.write_text(json.dumps({old: stale, old + "|lib:0123456789ab": stale}))
    cfg = autotune.autotune(vol, cache=str(path))
    assert len(tuned) == 1 and applied[-1]["uf_variant"] == 0 and cfg["key"].startswith(old)
    assert set(json.loads(path.read_text())) == {old, old + "|lib:0123456789ab", cfg["key"]}  # nothing of others' is lost
    # the same library: from the cache
    assert autotune.autotune(vol, cache=str(path))["key"] == cfg["key"] and len(tuned) == 1
    # other sources: made again
    monkeypatch.setattr(autotune, "kernels", lambda: "f" * 12)
    assert autotune.autotune(vol, cache=str(path))["key"] != cfg["key"] and len(tuned) == 2


def test_the_hash_covers_every_source():
    from paper_2606_04801_gb300 import autotune

    assert len(autotune.kernels()) == 12
    import os

    from paper_2606_04801_gb300 import build

    names = {os.path.basename(n) for n in build.CU + build.CPP + build.HEADERS}
    assert {f for f in os.listdir(build.CSRC) if f.endswith((".cu", ".cuh", ".h", ".cpp"))} <= names
