"""The native call module is optional: whatever stops its build, the library is
built all the same, no earlier module stays behind to be loaded, and the next
build makes it; a module that does not load, or is of another PyTorch, is left
out."""
import os
import stat

import pytest
import torch

from paper_2203_07673_gb300 import build, fmm


@pytest.fixture
def tree(tmp_path, monkeypatch):
    """A build folder with a library and a module of an earlier build, and a
    compiler that writes what it is asked for unless `fails` names a flag."""
    out = tmp_path / "_build"
    out.mkdir()
    lib, calls, cxx = out / "libfmm.so", out / "fmm_calls.so", tmp_path / "g++"
    lib.write_text("library")
    calls.write_text("earlier")

    def compiler(fails="never"):
        cxx.write_text("#!/bin/sh\nfor a in \"$@\"; do [ \"$a\" = \"%s\" ] && exit 1\n"
                       "[ \"$o\" = 1 ] && echo new > \"$a\"; o=0; [ \"$a\" = -o ] && o=1\ndone\n"
                       "exit 0\n" % fails)
        cxx.chmod(cxx.stat().st_mode | stat.S_IXUSR)
    compiler()
    monkeypatch.setattr(build, "OUT", str(out))
    monkeypatch.setattr(build, "LIB", str(lib))
    monkeypatch.setattr(build, "CALLS", str(calls))
    monkeypatch.setattr(build, "CXX", str(cxx))
    monkeypatch.setattr(build, "sources", lambda: [])
    return calls, compiler


@pytest.mark.parametrize("fails", ["-c", "-shared"])
def test_a_failed_step_leaves_no_module(tree, fails, capsys):
    calls, compiler = tree
    compiler(fails)
    assert os.path.exists(build.build_library())
    assert not calls.exists() and "not built" in capsys.readouterr().err
    compiler()
    build.build_library()
    assert calls.read_text() == "new\n"
    calls.write_text("kept")        # up to date: not built again
    build.build_library()
    assert calls.read_text() == "kept"


def test_no_compiler(tree, monkeypatch, capsys):
    calls, _ = tree
    monkeypatch.setattr(build, "CXX", "/nowhere/g++")
    assert os.path.exists(build.build_library())
    assert not calls.exists() and "not built" in capsys.readouterr().err


def test_no_pytorch(tree, monkeypatch, capsys):
    calls, _ = tree
    monkeypatch.setattr(build.importlib.util, "find_spec", lambda name: None)
    assert os.path.exists(build.build_library())
    assert not calls.exists() and "PyTorch is not installed" in capsys.readouterr().err


def test_a_module_that_does_not_load(tmp_path, monkeypatch):
    """The library loads without it, at the first call as at the second."""
    bad = tmp_path / "fmm_calls.so"
    bad.write_text("not a module")
    monkeypatch.setattr(fmm, "CALLS_PATH", str(bad))
    monkeypatch.setattr(fmm, "_lib", None)
    monkeypatch.setattr(fmm, "_calls", None)
    with pytest.warns(UserWarning, match="does not load"):
        assert fmm.lib().fmm_version() > 0
    assert fmm._calls is None and fmm.lib().fmm_version() > 0


def test_a_module_of_another_pytorch(monkeypatch):
    if not os.path.exists(fmm.CALLS_PATH):
        pytest.skip("the module is not built")
    assert fmm._load_calls() is not None
    monkeypatch.setattr(torch, "__version__", "1.0.0+cpu")
    with pytest.warns(UserWarning, match="built for PyTorch"):
        assert fmm._load_calls() is None
