"""The autotuner's cache key (no GPU): it names the library's sources, so that a result measured on other
kernels is not taken for the current ones."""
import json
import os
import shutil
import types

import pytest

torch = pytest.importorskip("torch")

import __graft_entry__ as entry


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


def _key(monkeypatch):
    from paper_2304_12597_gb300.autotune import plan_key

    monkeypatch.setattr(torch.cuda, "get_device_name", lambda device: "GPU")
    return plan_key(types.SimpleNamespace(dim=1, nx=511, ny=1, nt=256, batch=1, precision="mixed", device="cuda:0",
                                          desc=types.SimpleNamespace(alpha=0.0)))


def test_key_changes_with_the_sources(monkeypatch, tmp_path):
    from paper_2304_12597_gb300 import build

    before = _key(monkeypatch)
    assert _key(monkeypatch) == before
    other = tmp_path / "csrc"
    shutil.copytree(build.CSRC, other)
    monkeypatch.setattr(build, "CSRC", str(other))
    assert _key(monkeypatch) == before  # the same files elsewhere
    with open(os.path.join(other, "pint_chunk.cu"), "a") as f:
        f.write("// changed\n")
    assert _key(monkeypatch) != before


def test_results_of_an_unnamed_build_are_not_found(monkeypatch, tmp_path):
    from paper_2304_12597_gb300.autotune import _cache_load, _cache_store

    key = _key(monkeypatch)
    old = {k: v for k, v in json.loads(key).items() if k != "build"}
    path = str(tmp_path / "tuned.json")
    _cache_store(path, json.dumps(old, sort_keys=True), {"tune": {"pint_rows": 8}, "ms": 1.0, "default_ms": 2.0})
    assert len(old) == 8 and _cache_load(path).get(key) is None
