"""The native module of the binding: rebuilt for another torch or Python, and done without where it is missing or does not fit."""
import os
import warnings

import pytest

from paper_2607_17419_b200 import binding as kb
from paper_2607_17419_b200 import build as kbuild


@pytest.fixture(autouse=True)
def built(monkeypatch):
    kbuild.build()
    monkeypatch.setattr(kb, "_native", None)


def left_to_ctypes(match):
    with pytest.warns(UserWarning, match=match):
        mod = kb.native()
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        assert kb.native() is mod
    assert all(getattr(mod, f)(*range(12)) is NotImplemented for f in ("forward", "decode", "backward"))


def test_built_for_this_torch():
    assert not kbuild.needs_build() and kbuild.host_current()
    assert kb.native().__name__.endswith("_kata_torch")


def test_another_torch(monkeypatch):
    tag = kbuild.host_tag()
    monkeypatch.setattr(kbuild, "host_tag", lambda: tag.replace("torch 2", "torch 3"))
    assert kbuild.needs_build()
    left_to_ctypes("another torch")


def test_missing(monkeypatch, tmp_path):
    monkeypatch.setattr(kbuild, "HOST", str(tmp_path / "none.so"))
    assert kbuild.needs_build()
    left_to_ctypes("missing")


def test_does_not_load(monkeypatch):
    import builtins
    real = builtins.__import__

    def broken(name, globals=None, locals=None, fromlist=(), level=0):
        if "_kata_torch" in (fromlist or ()):
            raise ImportError("undefined symbol")
        return real(name, globals, locals, fromlist, level)

    monkeypatch.setattr(builtins, "__import__", broken)
    left_to_ctypes("undefined symbol")


@pytest.mark.parametrize("host", [["false"], ["/nonexistent/compiler"]])
def test_library_without_the_module(monkeypatch, tmp_path, host):
    """libkata.so needs nvcc alone: a failing build of the module is a warning, and leaves no old module behind."""
    nvcc = tmp_path / "nvcc"
    nvcc.write_text('#!/bin/sh\nwhile [ "$1" != -o ]; do shift; done\n: > "$2"\n')
    nvcc.chmod(0o755)
    monkeypatch.setattr(kbuild, "HERE", str(tmp_path))
    monkeypatch.setattr(kbuild, "LIB", str(tmp_path / "libkata.so"))
    monkeypatch.setattr(kbuild, "HOST", str(tmp_path / "_kata_torch.so"))
    monkeypatch.setattr(kbuild, "_nvcc", lambda: str(nvcc))
    monkeypatch.setattr(kbuild, "_host_command", lambda obj: host)
    (tmp_path / "_kata_torch.so").write_text("of another build")
    with pytest.warns(UserWarning, match="not built"):
        assert kbuild.build(force=True) == str(tmp_path / "libkata.so")
    assert os.path.exists(tmp_path / "libkata.so") and not os.path.exists(tmp_path / "_kata_torch.so")
