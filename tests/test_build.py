"""What makes the built files stale."""
import glob
import os
import time

import pytest

from paper_2202_13808_b200 import build


@pytest.mark.parametrize("pattern", ["*.cu", "*.cuh", "*.h", "../../include/*.h"])
def test_a_newer_source_or_header_makes_the_library_stale(monkeypatch, pattern):
    build.build()
    assert not build._stale()
    newer = sorted(glob.glob(os.path.join(build.CSRC, pattern)))
    assert newer
    stat = os.path.getmtime
    for changed in newer:
        monkeypatch.setattr(os.path, "getmtime", lambda p: time.time() + 60 if os.path.samefile(p, changed) else stat(p))
        assert build._stale(), changed
        monkeypatch.undo()


@pytest.mark.parametrize("changed", ["native.cpp", "layer_ops.h", "dropit.h", "version.py"])       # the last one: torch's
def test_a_newer_source_header_or_torch_rebuilds_the_binding(monkeypatch, changed):
    build.build()
    commands, stat = [], os.path.getmtime
    monkeypatch.setattr(build.subprocess, "run", lambda command, check: commands.append(command))
    monkeypatch.setattr(build.os, "replace", lambda src, dst: None)
    build._build_native(False)
    assert not commands
    monkeypatch.setattr(os.path, "getmtime", lambda p: time.time() + 60 if os.path.basename(p) == changed else stat(p))
    build._build_native(False)
    assert len(commands) == 1 and build.NATIVE_SRC in commands[0]
