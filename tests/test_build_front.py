"""What the build does with the front end's C++ nodes: left out where torch is not installed, made again for another
torch, and no obstacle to the C library when they do not compile.  Compilers are faked (each writes its command line to
its output)."""
import subprocess
import sys
from types import SimpleNamespace

import pytest
import torch

from paper_2402_17427_gb300 import _build
from paper_2402_17427_gb300 import rasterize as R


@pytest.fixture
def fake(monkeypatch, tmp_path):
    for name, path in (("LIB", "lib.so"), ("FRONT", "front.so"), ("OUT_DIR", "out")):
        monkeypatch.setattr(_build, name, str(tmp_path / path))
    monkeypatch.setattr(_build, "nvcc", lambda: "/nowhere/bin/nvcc")
    state = SimpleNamespace(made=[], fail=lambda cmd: False)

    def run(cmd, **_):
        if state.fail(cmd):
            return SimpleNamespace(returncode=1, stdout="", stderr="no")
        with open(cmd[cmd.index("-o") + 1], "w") as f:
            f.write(" ".join(cmd))
        state.made.append("front" if _build.FRONT_SRC in cmd else "link" if "-shared" in cmd else "object")
        return SimpleNamespace(returncode=0, stdout="", stderr="")
    monkeypatch.setattr(subprocess, "run", run)
    state.exists = lambda p: (tmp_path / p).exists()
    return state


def test_library_without_torch(fake, monkeypatch):
    monkeypatch.setitem(sys.modules, "torch", None)      # import torch raises ImportError
    _build.build()
    assert fake.exists("lib.so") and not fake.exists("front.so") and "front" not in fake.made
    fake.made.clear()
    _build.build()
    assert fake.made == []


def test_nodes_are_made_again_for_another_torch(fake, monkeypatch):
    _build.build()
    assert fake.made.count("front") == 1 and fake.made.count("link") == 1
    fake.made.clear()
    _build.build()
    assert fake.made == []
    monkeypatch.setattr(torch, "__version__", "0.0.1+other")
    monkeypatch.setattr(R, "_front_module", None)
    with pytest.raises(RuntimeError, match="another torch"):
        R._front()
    _build.build()
    assert fake.made == ["front"]


def test_library_stands_when_the_nodes_do_not_compile(fake, monkeypatch):
    fake.fail = lambda cmd: _build.FRONT_SRC in cmd
    with pytest.raises(RuntimeError):
        _build.build()
    assert fake.exists("lib.so")
    monkeypatch.setattr(R, "_front_module", None)
    assert R._front() is None      # rasterize() and l1_dssim_loss() take the nodes written in Python


def test_the_built_nodes_carry_what_they_were_made_for():
    _build.build()
    assert _build.front_matches(torch)
    assert R._front().Uses().value == 0
