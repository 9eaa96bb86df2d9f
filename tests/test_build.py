"""When the built libraries are built again (CPU only; nothing is compiled here)."""
import os

import pytest

from paper_2607_20507_gb300 import build


@pytest.fixture()
def built(tmp_path, monkeypatch):
    for name in ("LIB", "MARSHAL", "AGAINST"):
        path = tmp_path / name
        path.write_text(build._built_against() if name == "AGAINST" else "")
        monkeypatch.setattr(build, name, str(path))
    newest = max(os.path.getmtime(f) for f in build._inputs())
    for name in ("LIB", "MARSHAL"):
        os.utime(getattr(build, name), (newest + 1, newest + 1))
    return tmp_path


def test_up_to_date(built):
    assert not build.is_stale()


@pytest.mark.parametrize("name", ["LIB", "MARSHAL", "AGAINST"])
def test_missing(built, name):
    os.remove(getattr(build, name))
    assert build.is_stale()


def test_another_torch(built):
    with open(build.AGAINST, "a") as f:
        f.write("torch 0")
    assert build.is_stale()


def test_newer_source(built):
    os.utime(build.LIB, (0, 0))
    assert build.is_stale()
