"""A changed source or header makes the library stale, whichever it is."""
import os
import shutil

import pytest

from paper_2104_07097_gb300 import build


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(build.CSRC)
                                        if f.endswith((".cu", ".cuh", ".h"))))
def test_newer_input_is_seen(name, tmp_path, monkeypatch):
    csrc = tmp_path / "csrc"
    shutil.copytree(build.CSRC, csrc)
    later = build._inputs_mtime() + 1000.0
    os.utime(csrc / name, (later, later))
    monkeypatch.setattr(build, "CSRC", str(csrc))
    assert build._inputs_mtime() == later
