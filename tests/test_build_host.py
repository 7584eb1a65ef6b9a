"""The native half of the binding is rebuilt for another torch or interpreter, says what it misses, and its absence is
reported as a build that is missing. On the CPU; nothing here builds the library."""
import sys

import pytest

from paper_2312_05693_b200 import binding, build


def test_a_module_built_for_another_torch_is_stale(tmp_path, monkeypatch):
    module, tag = tmp_path / "_aq_host.so", tmp_path / "built_for"
    module.write_bytes(b"")
    monkeypatch.setattr(build, "HOST_LIB", str(module))
    monkeypatch.setattr(build, "HOST_TAG", str(tag))
    assert build._host_stale()                                   # nobody knows what it was built for
    tag.write_text(build._host_tag())
    assert not build._host_stale()
    tag.write_text(build._host_tag() + "x")
    assert build._host_stale()


def test_missing_headers_are_named(monkeypatch, tmp_path):
    monkeypatch.setattr(build.sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
    with pytest.raises(RuntimeError, match="Python.h"):
        build._build_host()


def test_the_compiler_is_the_environments(monkeypatch):
    seen = []
    monkeypatch.setenv("CXX", "another-compiler")
    monkeypatch.setattr(build.subprocess, "check_call", seen.append)
    monkeypatch.setattr(build.os, "replace", lambda a, b: (_ for _ in ()).throw(InterruptedError()))
    with pytest.raises(InterruptedError):
        build._build_host()
    assert seen[0][0] == "another-compiler"


def test_an_absent_module_is_reported_as_a_missing_build(monkeypatch):
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(binding, "load", lambda: None)
    monkeypatch.setitem(sys.modules, "paper_2312_05693_b200._aq_host", None)
    monkeypatch.delattr(sys.modules["paper_2312_05693_b200"], "_aq_host", raising=False)
    with pytest.raises(ImportError, match="paper_2312_05693_b200.build"):
        binding._host()
