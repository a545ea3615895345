"""A source newer than the library makes it stale, whichever kind of source it is."""
import os

import pytest

from paper_2510_12901_gb300 import _build


@pytest.mark.parametrize("ext", [".cu", ".cuh", ".h"])
def test_a_newer_source_makes_the_library_stale(monkeypatch, ext):
    monkeypatch.setattr(os.path, "exists", lambda p: True)
    monkeypatch.setattr(os.path, "getmtime", lambda p: 1.0)
    assert not _build._stale()
    monkeypatch.setattr(os.path, "getmtime", lambda p: 2.0 if p.endswith(ext) else 1.0)
    assert _build._stale()
