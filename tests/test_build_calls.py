"""The native call module is optional: whatever stops its build, the library is
built all the same, no earlier module stays behind to be loaded, and the next
build makes it."""
import os
import stat

import pytest

from paper_2203_07673_gb300 import build


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
