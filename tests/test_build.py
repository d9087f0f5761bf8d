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
