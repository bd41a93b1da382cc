"""The library is rebuilt when anything it is compiled from changes: sources, private headers (.h and .cuh) and the
public ones."""

import os

import pytest

from paper_2103_10380_gb300 import build

INCLUDE = os.path.join(build.ROOT, "include")
FILES = [os.path.join(d, f) for d in (build.CSRC, INCLUDE) for f in sorted(os.listdir(d))]


@pytest.mark.parametrize("changed", FILES, ids=os.path.basename)
def test_a_changed_file_is_newer_than_the_library(changed, monkeypatch):
    getmtime = os.path.getmtime
    monkeypatch.setattr(os.path, "getmtime",
                        lambda p: 1e12 if os.path.exists(p) and os.path.samefile(p, changed) else getmtime(p))
    assert build._deps_mtime() == 1e12
