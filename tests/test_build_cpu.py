"""The library is rebuilt when any file that it is compiled from is newer than it."""
import os

import pytest

from paper_2204_07716_gb300 import build


@pytest.mark.parametrize("sub,name", [("csrc", "a.cu"), ("csrc", "a.cpp"), ("csrc", "a.cuh"),
                                      ("csrc", "a.h"), ("include", "a.h")])
def test_newer_source_makes_the_library_stale(tmp_path, monkeypatch, sub, name):
    for d in ("csrc", "include"):
        (tmp_path / d).mkdir()
    lib, src = tmp_path / "lib.so", tmp_path / sub / name
    lib.write_text("")
    src.write_text("")
    monkeypatch.setattr(build, "CSRC", str(tmp_path / "csrc"))
    monkeypatch.setattr(build, "INCLUDE", str(tmp_path / "include"))
    os.utime(src, (1000, 1000))
    os.utime(lib, (2000, 2000))
    assert not build._stale(str(lib))
    os.utime(src, (3000, 3000))
    assert build._stale(str(lib))
