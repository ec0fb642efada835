"""What build.py builds, and when."""
import importlib.util
import os

import pytest

from paper_2309_06626_b200 import build


@pytest.fixture
def asked(monkeypatch, tmp_path):
    """build() with a library that is up to date and no extension: what it does about the latter."""
    done = []
    monkeypatch.setattr(build, "is_stale", lambda: False)
    monkeypatch.setattr(build, "EXT", str(tmp_path / "_asx_torch.so"))
    monkeypatch.setattr(build, "_build_ext", lambda: done.append("extension"))
    return done


def test_the_library_is_built_without_torch(asked, monkeypatch):
    found = importlib.util.find_spec
    assert build.build() == build.LIB and asked == ["extension"]
    monkeypatch.setattr(importlib.util, "find_spec", lambda name, *a: None if name == "torch" else found(name, *a))
    assert build.build() == build.LIB and asked == ["extension"]
