"""What makes a translation unit's object out of date (no compiler is run)."""
import os

import pytest

from paper_1910_01011_gb300 import build


@pytest.mark.parametrize("changed", ["a.cu", "b.h", "c.cuh", None])
def test_objects_depend_on_every_header(tmp_path, monkeypatch, changed):
    for f in ("a.cu", "b.h", "c.cuh", "a.cu.o"):
        (tmp_path / f).write_text("")
        os.utime(tmp_path / f, (2_000_000_000, 2_000_000_000))  # later than the public header
    monkeypatch.setattr(build, "CSRC", str(tmp_path))
    if changed:
        os.utime(tmp_path / changed, (2_000_000_010, 2_000_000_010))
    assert build._stale(str(tmp_path / "a.cu.o"), str(tmp_path / "a.cu")) == (changed is not None)
