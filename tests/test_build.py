"""What the in-tree build needs and when it is repeated (CPU only)."""
from __future__ import annotations

import ctypes
import sys

import pytest

from paper_2609_14636_gb300 import _build


@pytest.fixture
def tree(monkeypatch, tmp_path):
    """The build's results in an empty folder, of one source file."""
    monkeypatch.setattr(_build, "LIB", tmp_path / "libstride.so")
    monkeypatch.setattr(_build, "BUILD", tmp_path / "_build")
    monkeypatch.setattr(_build, "PKG", tmp_path)
    monkeypatch.setattr(_build, "sources", lambda: [_build.CSRC / "api.cu"])
    return tmp_path


def test_library_builds_without_torch(tree, monkeypatch):
    """A C caller's machine has nvcc and no torch."""
    monkeypatch.setitem(sys.modules, "torch", None)
    with pytest.warns(RuntimeWarning, match="native marshalling"):
        assert _build.build() == tree / "libstride.so"
    assert (tree / "libstride.so").exists() and not list(tree.glob("_binding*"))
    assert _build.up_to_date()


def test_calls_without_the_marshalling(monkeypatch):
    """Every entry point's general code takes the calls then."""
    import paper_2609_14636_gb300 as stride

    def fails(force=False):
        raise RuntimeError("no compiler")

    monkeypatch.setattr(stride, "_NATIVE", None)
    monkeypatch.setattr(_build, "build_binding", fails)
    with pytest.warns(RuntimeWarning, match="no compiler"):
        native = stride._native()
    assert all(getattr(native, fn)(1, 2, 3) is None for fn in stride._NATIVE_ENTRIES)
    assert isinstance(stride.lib(), ctypes.CDLL)


def test_marshalling_of_another_torch_or_interpreter(tree, monkeypatch):
    """One built for another torch or interpreter, whose layouts it holds, is not taken for this one's."""
    import torch

    built = []

    def compiler(cmd, **kw):  # stands for g++
        out = cmd[cmd.index("-o") + 1]
        built.append(out)
        open(out, "w").close()
        return _build.subprocess.CompletedProcess(cmd, 0, "", "")

    monkeypatch.setattr(_build.subprocess, "run", compiler)
    first = _build.build_binding()
    assert _build.build_binding() == first and len(built) == 1
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    second = _build.build_binding()
    monkeypatch.setattr(_build.sysconfig, "get_config_var", lambda name: "cpython-399")
    third = _build.build_binding()
    assert len({first, second, third}) == 3 and len(built) == 3
