"""The library without the binding's C++ part: where that cannot be built or loaded, the Python code stands in (csrc/binding.cpp)."""
import os
import shutil
import subprocess
import sys

import pytest

import paper_2407_12077_b200 as gf
from paper_2407_12077_b200 import _build


def test_a_file_that_cannot_be_loaded_is_done_without(tmp_path, monkeypatch):
    # (left by a torch it does not fit, or half copied)
    lib = gf.load_library()
    native = gf._native
    for content in (b"not a shared object", b""):
        path = tmp_path / "binding.so"
        path.write_bytes(content)
        monkeypatch.setattr(_build, "BINDING_PATH", str(path))
        monkeypatch.setattr(gf, "_native", None)
        gf._load_native(lib)
        assert gf._native is None
    monkeypatch.undo()
    assert gf._native is native


def test_a_compiler_that_fails_leaves_the_library_as_it_is(tmp_path):
    # a copy of the package whose CUDA library is built and whose C++ part is not, and a g++ that fails first on the path
    gf.load_library()
    root = os.path.dirname(os.path.dirname(os.path.abspath(gf.__file__)))
    shutil.copytree(os.path.dirname(gf.__file__), tmp_path / "paper_2407_12077_b200", ignore=shutil.ignore_patterns("_binding*", "__pycache__"))
    shutil.copytree(os.path.join(root, "include"), tmp_path / "include")
    gxx = tmp_path / "bin" / "g++"
    gxx.parent.mkdir()
    gxx.write_text("#!/bin/sh\necho no such header >&2\nexit 1\n")
    gxx.chmod(0o755)
    code = ("import warnings; warnings.simplefilter('always'); import paper_2407_12077_b200 as gf; gf.load_library(); "
            "print(gf.__file__, gf.version(), gf._native)")
    r = subprocess.run([sys.executable, "-c", code], cwd=tmp_path, env=dict(os.environ, PATH="%s:%s" % (gxx.parent, os.environ["PATH"])),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-500:]
    where, version, native = r.stdout.split()
    assert where.startswith(str(tmp_path)) and int(version) == gf.version() and native == "None"
    assert "no such header" in r.stderr                      # (said, not raised)
    assert not [f for f in os.listdir(tmp_path / "paper_2407_12077_b200") if f.startswith("_binding")]


def test_the_cuda_library_is_built_whatever_becomes_of_the_binding(monkeypatch):
    built = []

    def run(cmd, **kw):
        built.append(os.path.basename(cmd[0]))
        return subprocess.CompletedProcess(cmd, int(built[-1] == "g++"), "", "no such header")

    monkeypatch.setattr(_build.subprocess, "run", run)
    with pytest.warns(RuntimeWarning, match="no such header"):
        assert _build.build(force=True) == _build.LIB_PATH
    assert built == ["nvcc", "g++"]
