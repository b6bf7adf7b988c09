"""The build where the binding cannot be had, and a binding that was built against another torch."""
import subprocess
import sys
import types

import pytest

import paper_2509_24695_b200 as la
from paper_2509_24695_b200 import build


@pytest.fixture
def tree(tmp_path, monkeypatch):
    """A build of no kernels into a folder of its own."""
    monkeypatch.setattr(build, "sources", lambda: [])
    for name, file in (("LIB", "lib.so"), ("BINDING", "binding.so"), ("STAMP", "build/stamp")):
        monkeypatch.setattr(build, name, str(tmp_path / file))
    links = []

    def link(cmd):
        links.append(cmd)
        open(cmd[cmd.index("-o") + 1], "w").close()

    monkeypatch.setattr(subprocess, "check_call", link)
    return tmp_path, links


WORKS = lambda out: [sys.executable, "-c", f"open({out!r}, 'w').close()"]
FAILS = lambda out: [sys.executable, "-c", "raise SystemExit('no such header')"]


@pytest.mark.parametrize("command", [FAILS, lambda out: ["/nowhere/g++"], lambda out: None], ids=["fails", "no compiler", "no torch"])
def test_the_library_is_built_without_the_binding(tree, command, monkeypatch, capfd):
    folder, links = tree
    (folder / "binding.so").touch()   # of an earlier build
    monkeypatch.setattr(build, "_binding_command", command)
    assert build.build() == str(folder / "lib.so") and (folder / "lib.so").exists()
    assert not (folder / "binding.so").exists() and "warning" in capfd.readouterr().err
    assert build.build() and len(links) == 1                       # nothing to do
    monkeypatch.setattr(build, "_binding_command", WORKS)
    assert build.build(force=True) and (folder / "binding.so").exists() and len(links) == 2
    assert build.build() and len(links) == 2
    (folder / "binding.so").unlink()                               # lost: built again
    assert build.build() and (folder / "binding.so").exists() and len(links) == 3


@pytest.mark.parametrize("other", [{}, {"built_against": "1.0.0"}], ids=str)
def test_a_binding_of_another_torch_is_left_alone(other, monkeypatch):
    def bind(*args):
        raise AssertionError("bound")

    module = types.SimpleNamespace(bind=bind, **other)
    monkeypatch.setitem(sys.modules, la.__name__ + "._binding", module)
    monkeypatch.setattr(la, "_binding", module, raising=False)
    monkeypatch.setattr(la, "_fast", None)
    assert la._bind(None) is la._NoBinding
