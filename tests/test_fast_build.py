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


def test_the_library_builds_without_a_compiler_for_the_extension(monkeypatch, capsys):
    import __graft_entry__

    def no_compiler(force=False):
        raise FileNotFoundError("g++")

    monkeypatch.setattr(build, "build_fast", no_compiler)
    __graft_entry__.build()
    assert "g++" in capsys.readouterr().err


def test_the_extension_takes_the_toolkit_that_builds_the_library(monkeypatch, tmp_path):
    (tmp_path / "bin").mkdir()
    nvcc = tmp_path / "bin" / "nvcc"
    nvcc.write_text("")
    nvcc.chmod(0o755)
    seen = []
    monkeypatch.setenv("NVCC", str(nvcc))
    monkeypatch.setattr(build, "fast_so", lambda: tmp_path / "fast.so")
    monkeypatch.setattr(build.subprocess, "run", lambda cmd, check: seen.extend(cmd))
    monkeypatch.setattr(build.os, "replace", lambda a, b: None)
    build.build_fast()
    assert f"-I{tmp_path / 'include'}" in seen and "-I/usr/local/cuda/include" not in seen
