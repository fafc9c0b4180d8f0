"""Building and loading: the marshalling module is an extra, made for one Python and one torch."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2502_01941_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_library_is_built_without_the_marshalling_module(monkeypatch, tmp_path):
    """A host compiler that fails, a torch without headers: libshotkv.so all the same, and a warning."""
    made = []
    monkeypatch.setattr(build, "_build_cuda", lambda force, verbose: made.append("cuda") or build.LIB_PATH)
    monkeypatch.setattr(build, "marshal_path", lambda: str(tmp_path / "m.so"))
    monkeypatch.setenv("CXX", "false")
    with pytest.warns(UserWarning, match="ctypes"):
        assert build.build_library() == build.LIB_PATH
    assert made == ["cuda"] and not os.listdir(tmp_path)


def test_a_module_for_another_torch_is_not_the_one_loaded(monkeypatch):
    here = build.marshal_path()
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert build.marshal_path() != here
    assert build._stale(build.marshal_path(), [])


def test_importing_the_package_loads_no_native_code():
    """Only lib() does: a program that never calls the library has none of it in its process."""
    code = ("import paper_2502_01941_b200 as skv\n"
            "maps = lambda: {l.split('/')[-1].strip() for l in open('/proc/self/maps') if 'paper_2502_01941_b200' in l and '.so' in l}\n"
            "assert not maps(), maps()\n"
            "skv.lib()\n"
            "assert any('libshotkv' in m for m in maps()), maps()\n")
    subprocess.run([sys.executable, "-c", code], cwd=ROOT, check=True)
