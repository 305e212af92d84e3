"""The library is rebuilt when any file it is compiled from is newer."""
import os

import pytest

from paper_2402_11878_gb300 import build


@pytest.mark.parametrize("name", ["vqe_api.cu", "vqe_internal.h", "pass_core.cuh", "vqe.h"])
def test_every_source_counts(tmp_path, monkeypatch, name):
    for f in ("vqe_api.cu", "vqe_internal.h", "pass_core.cuh", "vqe.h"):
        (tmp_path / f).write_text("")
        os.utime(tmp_path / f, (100, 100))
    os.utime(tmp_path / name, (200, 200))
    monkeypatch.setattr(build, "CSRC", str(tmp_path))
    monkeypatch.setattr(build, "INCLUDE", str(tmp_path))
    assert build._deps_mtime() == 200
