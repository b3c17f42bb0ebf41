"""Loading the binding where its extension cannot be built: the numpy path serves, with a warning."""
import os
import shutil

import pytest

from paper_2609_35065_gb300 import build, kvs


@pytest.fixture
def nowhere(monkeypatch, tmp_path):
    """No extension yet, in a folder of its own."""
    monkeypatch.setattr(build, "OUT_DIR", str(tmp_path))
    monkeypatch.setattr(build, "PYCALL", str(tmp_path / "kvs_pycall.so"))
    return tmp_path


def _no_compiler(monkeypatch):
    which = shutil.which
    monkeypatch.setattr(build.shutil, "which", lambda c: None if c in ("gcc", "cc") else which(c))


def _unwritable(monkeypatch, folder):
    (folder / "file").write_text("")
    monkeypatch.setattr(build, "OUT_DIR", str(folder / "file" / "under"))
    monkeypatch.setattr(build, "PYCALL", str(folder / "file" / "under" / "kvs_pycall.so"))


def _broken_source(monkeypatch, folder):
    (folder / "bad.c").write_text("not C\n")
    monkeypatch.setattr(build, "PYCALL_SOURCE", str(folder / "bad.c"))


@pytest.mark.skipif(not build._has_python_headers(), reason="no Python headers")
def test_the_extension_builds_and_loads(nowhere):
    assert callable(build.load_pycall())


@pytest.mark.skipif(not build._has_python_headers(), reason="no Python headers")
@pytest.mark.parametrize("cause", ["no_compiler", "unwritable", "broken_source"])
def test_an_extension_that_cannot_be_built_is_done_without(monkeypatch, nowhere, cause):
    if cause == "no_compiler":
        _no_compiler(monkeypatch)
    elif cause == "unwritable":
        _unwritable(monkeypatch, nowhere)
    else:
        _broken_source(monkeypatch, nowhere)
    with pytest.warns(RuntimeWarning, match="cannot be built"):
        assert build.load_pycall() is None


def test_a_library_that_is_there_loads_without_the_extension(monkeypatch, tmp_path):
    kvs.lib()
    monkeypatch.setattr(build, "PYCALL", str(tmp_path / "kvs_pycall.so"))
    monkeypatch.setattr(kvs, "_lib", None)
    monkeypatch.setattr(kvs, "_pycall", None)
    monkeypatch.setattr(build, "_has_python_headers", lambda: True)
    monkeypatch.setenv("KVS_LIBRARY", kvs.lib_path())
    _no_compiler(monkeypatch)
    with pytest.warns(RuntimeWarning, match="cannot be built"):
        assert kvs.lib().kvs_last_error() is not None
    assert kvs._pycall is None


def test_an_older_extension_is_not_used_when_it_cannot_be_rebuilt(monkeypatch, nowhere):
    if build._has_python_headers():
        build.build_pycall()
    else:
        open(build.PYCALL, "w").close()
    os.utime(build.PYCALL, (1, 1))
    monkeypatch.setattr(build, "_has_python_headers", lambda: False)
    assert build.load_pycall() is None


def test_a_file_that_is_no_extension_is_not_used(nowhere):
    with open(build.PYCALL, "w") as f:
        f.write("not a shared object")
    with pytest.warns(RuntimeWarning, match="cannot be loaded"):
        assert build.load_pycall() is None
