"""The decode calls' native marshalling is loaded only where it was built for the Python, the torch and the source at hand."""
import sysconfig

import pytest
import torch

from paper_2602_01744_b200 import api, build


def test_what_was_built_for_something_else_is_not_found(monkeypatch, tmp_path):
    places = {build.fast_so()}
    with monkeypatch.context() as m:
        m.setattr(torch, "__version__", "0.0.0")
        places.add(build.fast_so())
    with monkeypatch.context() as m:
        m.setattr(sysconfig, "get_config_var", lambda name: "cpython-000")
        places.add(build.fast_so())
    source = tmp_path / "fastcall.cpp"
    source.write_text(build.FAST_SOURCE.read_text() + "\n")
    with monkeypatch.context() as m:
        m.setattr(build, "FAST_SOURCE", source)
        places.add(build.fast_so())
    assert len(places) == 4


def test_without_a_current_build_the_python_path_serves_and_says_so(monkeypatch):
    L = api.lib()
    monkeypatch.setattr(api, "_fast", None)

    def no_compiler(force=False):
        raise FileNotFoundError("g++")

    monkeypatch.setattr(build, "build_fast", no_compiler)
    with pytest.warns(RuntimeWarning, match="Python path"):
        api._load_fast(L)
    assert api._fast is None


def test_the_extension_loads():
    api.lib()
    assert api._fast is not None
