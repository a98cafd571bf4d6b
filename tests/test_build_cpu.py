"""When build() compiles again (the compilers themselves are not run here)."""
import os

import pytest

from paper_2604_07853_b200 import build


@pytest.fixture
def built(tmp_path, monkeypatch):
    """A tree in which both files are newer than their sources; yields the list of what build() compiles."""
    calls = []
    for name in ("LIB", "NATIVE", "NATIVE_KEY"):
        monkeypatch.setattr(build, name, str(tmp_path / name))
        (tmp_path / name).write_text("")
    monkeypatch.setattr(build, "_build_library", lambda verbose: calls.append("library"))
    monkeypatch.setattr(build, "_build_native", lambda: calls.append("native"))
    (tmp_path / "NATIVE_KEY").write_text(build.native_key())
    yield calls


def test_nothing_to_do(built):
    build.build()
    assert built == []


def test_other_torch_or_python_builds_the_marshalling_again(built, monkeypatch):
    monkeypatch.setattr(build, "native_key", lambda: "cpython-399\n/usr/include/python3.99\n9.9\n/elsewhere/torch")
    build.build()
    assert built == ["native"]


def test_a_file_of_unknown_origin_is_built_again(built):
    os.remove(build.NATIVE_KEY)
    build.build()
    assert built == ["native"]
