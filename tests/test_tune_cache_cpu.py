"""The autotuner's on-disk choices belong to the kernels they were timed on."""
import json
from types import SimpleNamespace

import pytest

from paper_2010_12117_gb300 import tune


class FakeBatch:
    """Orders 5 and 24, one million items each; records what it is told."""

    def __init__(self):
        self.info = SimpleNamespace(items={5: 1 << 20, 24: 1 << 20})
        self.told = {}

    def orders(self):
        return [5, 24]

    def set_mode(self, n, mode):
        self.told[n] = [mode]

    def set_launch(self, n, threads):
        self.told[n].append(threads)


@pytest.fixture
def cache(monkeypatch, tmp_path):
    monkeypatch.setattr(tune, "CACHE_DIR", str(tmp_path))
    monkeypatch.setattr(tune, "CACHE", str(tmp_path / "batch_launch.json"))
    monkeypatch.setattr(tune.torch.cuda, "get_device_name", lambda *a: "NVIDIA GB300")
    return tmp_path / "batch_launch.json"


CHOICES = {"NVIDIA_GB300/n24/items2^20": {"mode": 0, "threads": 64, "ms": 1.0}}


def test_choices_of_this_build_are_applied(cache):
    tune._save(CHOICES)
    b = FakeBatch()
    assert set(tune.apply_cached(b)) == {24}
    assert b.told == {24: [0, 64]}


def test_choices_of_another_build_are_not_applied(cache, monkeypatch):
    cache.write_text(json.dumps(CHOICES))  # a file that names no build
    b = FakeBatch()
    assert tune.apply_cached(b) == {} and b.told == {}
    tune._save(CHOICES)
    monkeypatch.setattr(tune, "source_id", lambda: "other kernels")
    assert tune.apply_cached(b) == {} and b.told == {}
    tune._save({})  # replaces what the other build left
    assert json.loads(cache.read_text()) == {"build": "other kernels", "choices": {}}


def test_unreadable_cache_is_empty(cache):
    for text in ("", "{", "[]", '{"build": "x"}'):
        cache.write_text(text)
        assert tune.apply_cached(FakeBatch()) == {}
