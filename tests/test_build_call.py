"""The native call from Python belongs to one interpreter and one torch, and is not what the library depends on (no GPU)."""
import importlib.metadata
import os
import sysconfig

import pytest

from paper_2502_01662_b200 import binding, build


def test_the_module_is_named_after_what_it_was_built_for(monkeypatch):
    path = build.call_path()
    assert sysconfig.get_config_var("SOABI") in path and importlib.metadata.version("torch") in path
    build.build_call()
    assert os.path.exists(path) and not build.call_needs_build()
    monkeypatch.setattr(importlib.metadata, "version", lambda name: "0.0.1")
    assert build.call_path() != path and build.call_needs_build()


def test_a_new_source_makes_it_stale(monkeypatch):
    build.build_call()
    newer = os.path.getmtime(build.call_path()) + 10
    before = os.path.getmtime
    monkeypatch.setattr(os.path, "getmtime", lambda f: newer if f == build.CALL_SOURCE else before(f))
    assert build.call_needs_build()
    assert build.CALL_SOURCE not in build.dependencies()      # (the CUDA library does not hang on it)


@pytest.mark.parametrize("what", ["no compiler", "not a module"])
def test_without_it_calls_go_the_long_way(monkeypatch, tmp_path, what):
    broken = tmp_path / "_call.so"
    broken.write_bytes(b"nothing")

    def build_call(force=False):
        if what == "no compiler":
            raise RuntimeError("g++ failed")
        return str(broken)

    monkeypatch.setattr(build, "build_call", build_call)
    monkeypatch.setattr(binding, "_call", None)
    with pytest.warns(RuntimeWarning, match="the long way"):
        assert binding.load_call() is None
    assert binding.load_call() is None                         # (said once)


def test_it_opens():
    assert callable(binding.load_call().run)
