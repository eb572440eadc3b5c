"""csrc/network.cpp is optional: what does not compile, or was built for another torch or Python, is left out and the Python code takes its place."""
import os
import subprocess
import sys

import pytest

from paper_2311_14272_b200 import build as build_mod

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _python(code):
    return subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)


def test_the_module_says_what_it_was_built_for():
    build_mod.build()
    if not (build_mod.HAVE_PYTHON_H and build_mod.torch_dir()):
        pytest.skip("no headers")
    out = _python("from paper_2311_14272_b200 import binding as B\nassert B._bind_network() and B._network.built_for.endswith(' %d.%d')\nprint('bound', B._network.built_for)"
                  % sys.version_info[:2])
    assert out.returncode == 0 and "bound" in out.stdout, out.stderr


@pytest.mark.parametrize("built_for", [None, "1.0.0 3.12", "2.11.0 2.7"])
def test_a_module_for_other_libraries_is_not_used(built_for):
    code = """
import sys, types
other = types.ModuleType("paper_2311_14272_b200._network")
other.bind = lambda address: calls.append(address)
calls, built_for = [], %r
if built_for:
    other.built_for = built_for
import paper_2311_14272_b200
sys.modules["paper_2311_14272_b200._network"] = paper_2311_14272_b200._network = other
from paper_2311_14272_b200 import binding as B
assert B._bind_network() is False and B._bind_network() is False and B._network is False and not calls
print("left out")
""" % (built_for,)
    build_mod.build()
    out = _python(code)
    assert out.returncode == 0 and "left out" in out.stdout, out.stderr


def test_a_failed_compile_is_not_an_error(tmp_path, monkeypatch, capsys):
    if not (build_mod.HAVE_PYTHON_H and build_mod.torch_dir()):
        pytest.skip("no headers")
    compiler = tmp_path / "cxx"
    compiler.write_text('#!/bin/sh\nfor a; do case $a in *network.cpp) exit 1;; esac; done\nexec ${REAL_CXX:-g++} "$@"\n')
    compiler.chmod(0o755)
    old = tmp_path / "_network.so"
    old.write_bytes(b"of other sources")
    monkeypatch.setenv("CXX", str(compiler))
    monkeypatch.setattr(build_mod, "NETWORK", str(old))
    monkeypatch.setattr(build_mod, "_stale", lambda: False)
    assert build_mod.build_network(force=True) is False and not old.exists() and "does not compile" in capsys.readouterr().err
    assert build_mod.build() == build_mod.LIB and not old.exists()        # (tried again, and left out again)
    assert os.listdir(tmp_path) == ["cxx"]
    monkeypatch.setenv("CXX", str(tmp_path / "no_such_compiler"))
    assert build_mod.build_network(force=True) is False


def test_newer_headers_build_it_again(tmp_path, monkeypatch):
    if not (build_mod.HAVE_PYTHON_H and build_mod.torch_dir()):
        pytest.skip("no headers")
    where = tmp_path / "torch"
    header = where / "include" / "torch" / "csrc" / "autograd" / "python_variable.h"
    header.parent.mkdir(parents=True)
    header.write_text("")
    built = tmp_path / "_network.so"
    built.write_bytes(b"")
    compiled = []

    def compile_(cmd):
        compiled.append(cmd)
        open(cmd[cmd.index("-o") + 1], "wb").close()

    monkeypatch.setattr(build_mod, "torch_dir", lambda: str(where))
    monkeypatch.setattr(build_mod, "NETWORK", str(built))
    monkeypatch.setattr(build_mod.subprocess, "check_call", compile_)
    now = os.path.getmtime(built)
    os.utime(header, (now - 10, now - 10))
    os.utime(built, (now + 1000, now + 1000))
    assert build_mod.build_network() and not compiled
    os.utime(header, (now + 2000, now + 2000))
    assert build_mod.build_network() and len(compiled) == 1
