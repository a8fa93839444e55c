"""The build's rule for compiling again: a change of any header, .h or .cuh, makes every object stale."""
import os

import pytest

from paper_1910_09534_gb300 import build


@pytest.mark.parametrize("name", [f for f in sorted(os.listdir(build.CSRC)) if f.endswith((".h", ".cuh"))])
def test_newer_header_makes_objects_stale(name, tmp_path, monkeypatch):
    for f in os.listdir(build.CSRC):
        (tmp_path / f).write_text("")
        os.utime(tmp_path / f, (1e9, 1e9))
    (tmp_path / "sycsim.h").write_text("")
    os.utime(tmp_path / "sycsim.h", (1e9, 1e9))
    monkeypatch.setattr(build, "CSRC", str(tmp_path))
    monkeypatch.setattr(build, "INCLUDE", str(tmp_path))
    os.utime(tmp_path / name, (2e9, 2e9))
    assert build._headers_mtime() == 2e9
