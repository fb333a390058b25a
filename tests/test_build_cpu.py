"""When the extension over torch tensors is compiled again: it is bound to the C++ interfaces of Python and torch and to boda.h."""
import os
import sys

import pytest

from paper_1606_00094_b200 import build


def test_the_extension_belongs_to_one_python_and_one_torch(monkeypatch):
    here = build.build_calls()
    assert os.path.exists(here) and not build.calls_stale()
    assert sys.implementation.cache_tag in os.path.basename(here)
    monkeypatch.setattr(build.importlib.metadata, "version", lambda name: "9.9.9")
    assert build.calls_path() != here and build.calls_stale()

    def missing(name):
        raise build.importlib.metadata.PackageNotFoundError(name)
    monkeypatch.setattr(build.importlib.metadata, "version", missing)
    assert build.calls_path() is None and not build.calls_stale() and build.build_calls() is None


@pytest.mark.parametrize("name", ["CALLS_SRC", "CALLS_HEADER"])
def test_the_extension_is_stale_once_its_source_or_the_header_is_newer(name, tmp_path, monkeypatch):
    here = build.build_calls()
    newer = tmp_path / "newer"
    newer.write_text("")
    os.utime(newer, (os.path.getmtime(here) + 10,) * 2)
    monkeypatch.setattr(build, name, str(newer))
    assert build.calls_stale()


def test_one_extension_is_kept():
    build.build_calls()
    assert [n for n in os.listdir(os.path.dirname(build.__file__)) if n.startswith("_torch_calls") and n.endswith(".so")] == [os.path.basename(build.calls_path())]
