"""The library without the binding's C++ part: where that cannot be built or loaded, the Python code stands in (csrc/binding.cpp)."""
import os
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
