"""The build recompiles an object file when anything it was made from is newer."""
import os

import pytest

from paper_2102_06248_gb300 import build as B


@pytest.mark.parametrize("touched", ["solver.cu", "sim.h", "stream.cuh", "fempic.h"])
def test_object_is_stale_after_any_of_its_sources_changed(tmp_path, monkeypatch, touched):
    csrc, include = tmp_path / "csrc", tmp_path / "include"
    csrc.mkdir(), include.mkdir()
    files = {name: (include if name == "fempic.h" else csrc) / name
             for name in ("solver.cu", "sim.h", "stream.cuh", "fempic.h")}
    obj = tmp_path / "solver.o"
    for k, f in enumerate([*files.values(), obj]):
        f.write_text("")
        os.utime(f, (1000 + k, 1000 + k))
    monkeypatch.setattr(B, "CSRC", str(csrc))
    monkeypatch.setattr(B, "INCLUDE", str(include))
    assert not B._stale(str(obj), str(files["solver.cu"]))
    os.utime(files[touched], (2000, 2000))
    assert B._stale(str(obj), str(files["solver.cu"]))
