"""Host tests of the build: the library needs nvcc alone, the native part of the binding is left out where it cannot be compiled."""
import importlib.util
import os
import shutil
import sys
import warnings

import pytest

PACKAGE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_06564_b200")


def _tool(path, body):
    path.write_text("#!/bin/sh\n" + body)
    path.chmod(0o755)
    return str(path)


WRITES_ITS_OUTPUT = 'while [ $# -gt 0 ]; do if [ "$1" = -o ]; then echo made > "$2"; fi; shift; done\n'


@pytest.fixture
def tree(tmp_path, monkeypatch):
    """build.py in a package of its own, with one source of each kind and an nvcc that only writes its output."""
    package = tmp_path / "package"
    (package / "csrc").mkdir(parents=True)
    (tmp_path / "include").mkdir()
    for name in ("csrc/one.cu", "csrc/calls.cpp", "../include/trdq.h"):
        (package / name).write_text("")
    shutil.copy(os.path.join(PACKAGE, "build.py"), package)
    monkeypatch.setenv("NVCC", _tool(tmp_path / "nvcc", WRITES_ITS_OUTPUT))
    monkeypatch.setenv("CXX", _tool(tmp_path / "cxx", WRITES_ITS_OUTPUT))
    return package


def _load(package):
    spec = importlib.util.spec_from_file_location("build_under_test", package / "build.py")
    module = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(module)
    return module


def test_both_are_built(tree):
    build = _load(tree)
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        assert build.build() == build.LIB
    assert os.path.exists(build.LIB) and os.path.exists(build.calls_path())
    os.remove(build.calls_path())
    build.build()   # the library is up to date, the calls are not
    assert os.path.exists(build.calls_path())


@pytest.mark.parametrize("missing", ["torch", "compiler", "compiler fails"])
def test_the_library_does_not_need_what_the_native_calls_need(tree, tmp_path, monkeypatch, missing):
    build = _load(tree)
    build.build()
    before = os.path.getmtime(build.LIB)
    calls = build.calls_path()
    if missing == "torch":
        monkeypatch.setitem(sys.modules, "torch", None)   # importing it raises ImportError
    else:
        monkeypatch.setenv("CXX", str(tmp_path / "nowhere") if missing == "compiler" else _tool(tmp_path / "fails", "exit 1\n"))
    os.remove(build.LIB)
    os.utime(calls, (1, 1))
    with pytest.warns(UserWarning, match="native calls"):
        assert build.build(force=True) == build.LIB
    assert os.path.getmtime(build.LIB) >= before
    assert not os.path.exists(calls)   # the one made from other sources is gone
    with pytest.warns(UserWarning, match="native calls"):
        assert build.build() == build.LIB    # nothing to do for the library


def test_a_failing_nvcc_raises(tree, tmp_path, monkeypatch):
    monkeypatch.setenv("NVCC", _tool(tmp_path / "fails", "exit 1\n"))
    with pytest.raises(RuntimeError, match="failed"):
        _load(tree).build()


def test_headers_of_an_nvcc_on_the_path(tree, tmp_path, monkeypatch):
    bin_ = tmp_path / "toolkit" / "bin"
    bin_.mkdir(parents=True)
    _tool(bin_ / "nvcc", WRITES_ITS_OUTPUT)
    monkeypatch.setenv("PATH", str(bin_), prepend=os.pathsep)
    monkeypatch.setenv("NVCC", "nvcc")
    assert f"-I{tmp_path / 'toolkit' / 'include'}" in _load(tree)._calls_command("out.so")


def test_another_torch_has_native_calls_of_its_own(tree, monkeypatch):
    import torch
    build = _load(tree)
    build.build()
    first = build.calls_path()
    monkeypatch.setattr(torch, "__version__", "0.0.0+other")
    assert build.calls_path() != first and not os.path.exists(build.calls_path())
    build.build()
    assert os.path.exists(build.calls_path()) and os.path.exists(first)
    os.utime(first, (1, 1))   # older than the sources: of no use to either
    build.build()
    assert os.path.exists(build.calls_path()) and not os.path.exists(first)


def test_native_calls_made_for_another_torch_are_not_loaded(monkeypatch):
    import torch
    from paper_2503_06564_b200 import trdq
    monkeypatch.setattr(trdq, "_native", None)
    monkeypatch.setattr(torch, "__version__", "0.0.0+other")
    with pytest.warns(UserWarning, match="native calls"):
        assert trdq._calls().rotate_quantize(None, 128, 0, None, None, None) is None
    assert type(trdq._native) is trdq._GeneralWay
    monkeypatch.undo()
    monkeypatch.setattr(trdq, "_native", None)
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        assert type(trdq._calls()) is not trdq._GeneralWay
