"""The build recompiles when a header changes, device headers (.cuh) among
them (CPU)."""
import os

import pytest

from paper_2502_10907_gb300 import build as B


@pytest.mark.parametrize("name", ["stream_plan.h", "kernel64.cuh", "pair_tile.cuh"])
def test_headers_count(name, tmp_path, monkeypatch):
    src = tmp_path / "csrc"
    inc = tmp_path / "include"
    src.mkdir()
    inc.mkdir()
    for d, f in ((src, "common.h"), (src, name), (inc, "mtf.h")):
        (d / f).write_text("")
        os.utime(d / f, (1000, 1000))
    monkeypatch.setattr(B, "SRC", str(src))
    monkeypatch.setattr(B, "ROOT", str(tmp_path))
    assert B._headers_mtime() == 1000
    os.utime(src / name, (2000, 2000))
    assert B._headers_mtime() == 2000
