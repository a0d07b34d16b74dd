"""The build: the C library is built by itself, whatever becomes of the Python module beside it."""
import subprocess
import sys

import pytest
import torch

from paper_2110_09195_b200 import build


def test_the_library_is_built_without_torch(monkeypatch, tmp_path, capfd):
    monkeypatch.setattr(build, "FAST", tmp_path / "_snn_fast.so")
    monkeypatch.setitem(sys.modules, "torch", None)   # importing it raises
    assert build.build() == build.LIB and build.LIB.exists()
    assert "_snn_fast.so was not built" in capfd.readouterr().err
    with pytest.raises(ImportError):
        build.build_fast()


def test_the_library_is_built_where_the_module_cannot_be(monkeypatch, tmp_path, capfd):
    monkeypatch.setattr(build, "FAST", tmp_path / "_snn_fast.so")
    for compiler in ("/bin/false", str(tmp_path / "no-such-compiler")):
        monkeypatch.setenv("CXX", compiler)
        assert build.build() == build.LIB and build.LIB.exists()
        assert "_snn_fast.so was not built" in capfd.readouterr().err
        with pytest.raises((RuntimeError, OSError)):
            build.build_fast()
    assert not build.FAST.exists()


def test_the_module_is_built_anew_for_another_torch(monkeypatch):
    build.build_fast()
    commands = []
    monkeypatch.setattr(subprocess, "run", lambda cmd, **_: commands.append(cmd) or subprocess.CompletedProcess(cmd, 1, "", ""))
    build.build_fast()
    assert not commands   # up to date
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    with pytest.raises(RuntimeError):
        build.build_fast()
    assert len(commands) == 1 and any("0.0.1" in a for a in commands[0])
