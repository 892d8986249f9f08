"""The in-tree build takes a header that a source includes as a reason to recompile."""
import glob
import os
import re
import shutil

import pytest

from paper_2510_02135_gb300 import _build


def _included():
    names = set()
    for f in glob.glob(os.path.join(_build.CSRC, "*")):
        if f.endswith((".cu", ".cuh", ".h")):
            with open(f) as src:
                names.update(re.findall(r'^#include "([^"/]+)"', src.read(), re.M))
    return sorted(names)


@pytest.mark.parametrize("name", _included())
def test_newer_header_is_seen(tmp_path, monkeypatch, name):
    csrc = tmp_path / "csrc"
    shutil.copytree(_build.CSRC, csrc)
    for f in csrc.iterdir():
        os.utime(f, (1000, 1000))
    os.utime(csrc / name, (2000, 2000))
    monkeypatch.setattr(_build, "CSRC", str(csrc))
    monkeypatch.setattr(_build, "INCLUDE", str(tmp_path))
    assert _build._headers_mtime() == 2000
