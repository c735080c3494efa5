"""The library is rebuilt when its sources or its build flags are newer."""
import os

import pytest

from paper_1811_04156_gb300 import build


@pytest.mark.parametrize("newer", ["source", "flags", "nothing"])
def test_up_to_date_sees_sources_and_flags(monkeypatch, tmp_path, newer):
    flags = os.path.getmtime(build.__file__)  # the flags stand in build.py itself
    source, lib = tmp_path / "a.cu", tmp_path / "lib.so"
    source.write_text("")
    lib.write_text("")
    monkeypatch.setattr(build, "CSRC", str(tmp_path))
    monkeypatch.setattr(build, "INCLUDE", str(tmp_path))
    monkeypatch.setattr(build, "LIB", str(lib))
    built = flags + (-10 if newer == "flags" else 10)
    os.utime(lib, (built, built))
    edited = built + (5 if newer == "source" else -5)
    os.utime(source, (edited, edited))
    assert build.up_to_date() == (newer == "nothing")
