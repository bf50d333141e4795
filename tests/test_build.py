"""The build on the CPU: the library does not depend on the binding's native calls."""
import ctypes
import os

import pytest

from paper_2503_18339_b200 import build


@pytest.fixture
def elsewhere(monkeypatch, tmp_path):
    """The library is up to date, the native calls would be built into a folder of their own."""
    build.build()
    monkeypatch.setattr(build, "HOST", str(tmp_path / "_host.so"))
    return tmp_path


def library_after(capfd):
    assert build.build() == build.LIB
    assert ctypes.CDLL(build.LIB).granq_status_string is not None
    assert not os.path.exists(build.HOST)
    assert len([line for line in capfd.readouterr().err.splitlines() if line.startswith("_host.so has not been built")]) == 1


def test_library_without_a_compiler_for_the_native_calls(elsewhere, monkeypatch, capfd):
    monkeypatch.setenv("CXX", "false")
    library_after(capfd)


def test_library_without_torch(elsewhere, monkeypatch, capfd):
    monkeypatch.setattr(build.importlib.util, "find_spec", lambda name: None)
    library_after(capfd)


def test_native_calls_of_an_older_source_do_not_stay(elsewhere, monkeypatch, capfd):
    with open(build.HOST, "w") as f:
        f.write("old")
    os.utime(build.HOST, (0, 0))
    monkeypatch.setenv("CXX", "false")
    library_after(capfd)
