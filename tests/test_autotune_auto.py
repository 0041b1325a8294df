"""The tuner never returns a kernel slower than the library's own choice: AUTO is among what it times, and answers stored
before it was are not used.  On the CPU, with a fake device and fake timings."""
import json
import types

import pytest

import paper_2402_06415_gb300 as ising
from paper_2402_06415_gb300 import autotune

torch = pytest.importorskip("torch")


class _FakeLattice:
    def __init__(self, *a, **k):
        pass

    def __enter__(self):
        return self

    def __exit__(self, *a):
        pass


@pytest.fixture
def fake(monkeypatch, tmp_path):
    props = types.SimpleNamespace(name="GPU", multi_processor_count=152)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: None)
    monkeypatch.setattr(torch.cuda, "get_device_properties", lambda d: props)
    monkeypatch.setattr(autotune.B, "Lattice", _FakeLattice)
    path = tmp_path / "tune.json"
    monkeypatch.setenv("ISING_TUNE_CACHE", str(path))
    return path


@pytest.mark.parametrize("L", [256, 1000, 2048])
def test_auto_is_timed_and_wins_where_it_is_the_fastest(fake, monkeypatch, L):
    speed = {ising.ISING_KERNEL_AUTO: 1600.0, ising.ISING_KERNEL_HALF: 115.0, ising.ISING_KERNEL_TILED: 800.0}
    monkeypatch.setattr(autotune, "time_config", lambda lat, cfg, *a, **k: speed[cfg["kernel"]])
    res = autotune.tune(L)
    assert res["config"]["kernel"] == ising.ISING_KERNEL_AUTO
    assert sum(r["kernel"] == ising.ISING_KERNEL_AUTO for r in res["table"]) == 1
    assert autotune.tune(L) == res  # from the cache


def test_a_faster_shape_still_beats_auto(fake, monkeypatch):
    monkeypatch.setattr(autotune, "time_config", lambda lat, cfg, *a, **k: float(cfg["tile_rows"]))
    assert autotune.tune(16384)["config"]["kernel"] == ising.ISING_KERNEL_TILED


def test_answers_of_the_earlier_candidates_are_not_used(fake, monkeypatch):
    slow = {"config": {"kernel": ising.ISING_KERNEL_HALF, "k": 1, "tile_rows": 1, "tile_words": 4}, "flips_per_ns": 115.0,
            "table": []}
    fake.write_text(json.dumps({"GPU|152|L=1000|layout=1": slow}))
    monkeypatch.setattr(autotune, "time_config",
                        lambda lat, cfg, *a, **k: 2.0 if cfg["kernel"] == ising.ISING_KERNEL_AUTO else 1.0)
    assert autotune.tune(1000)["config"]["kernel"] == ising.ISING_KERNEL_AUTO
