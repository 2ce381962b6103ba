"""The library is rebuilt when any file that its translation units are made of is newer than it."""
import os

import pytest

from paper_1211_0585_gb300 import build as B


@pytest.mark.parametrize("name", ["a.cu", "a.cuh", "a.h"])
def test_newer_source_makes_the_library_stale(tmp_path, monkeypatch, name):
    lib, src = tmp_path / "libwf.so", tmp_path / name
    src.write_text("")
    lib.write_text("")
    os.utime(src, (1000, 1000))
    os.utime(lib, (2000, 2000))
    monkeypatch.setattr(B, "LIB", str(lib))
    monkeypatch.setattr(B, "CSRC", str(tmp_path))
    monkeypatch.setattr(B, "INCLUDE", str(tmp_path / "include"))
    assert not B._stale()
    os.utime(src, (3000, 3000))
    assert B._stale()
