"""What build.py builds, and when."""
import importlib.metadata
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
    monkeypatch.setattr(build, "EXT_FOR", str(tmp_path / "_asx_torch.built_for"))
    monkeypatch.setattr(build, "_build_ext", lambda: done.append("extension"))
    return done


def test_the_library_is_built_without_torch(asked, monkeypatch):
    found = importlib.util.find_spec
    assert build.build() == build.LIB and asked == ["extension"]
    monkeypatch.setattr(importlib.util, "find_spec", lambda name, *a: None if name == "torch" else found(name, *a))
    assert build.build() == build.LIB and asked == ["extension"]


def test_the_extension_is_built_anew_for_another_torch(asked, monkeypatch):
    def put():
        open(build.EXT, "w").close()
        with open(build.EXT_FOR, "w") as f:
            f.write(build._ext_target())
    put()
    build.build()
    assert asked == []
    version = importlib.metadata.version
    with monkeypatch.context() as m:
        m.setattr(importlib.metadata, "version", lambda name: "99.0" if name == "torch" else version(name))
        build.build()
        assert asked == ["extension"]
        put()
        build.build()
        assert asked == ["extension"]
    build.build()
    assert asked == ["extension"] * 2
    put()
    os.remove(build.EXT_FOR)                     # one that does not say what it was built for
    build.build()
    assert asked == ["extension"] * 3
