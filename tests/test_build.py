"""What is built without what: the library needs nvcc alone, the extension module a C compiler and Python's headers."""
import os

import pytest

from paper_2409_13761_b200 import build


@pytest.fixture
def commands(monkeypatch):
    """Nothing is up to date, no command is run: what would have been is recorded; C compilers fail."""
    seen = []

    def run(cmd, check):
        seen.append(cmd)
        if os.path.basename(cmd[0]) in ("gcc", "cc"):
            raise build.subprocess.CalledProcessError(1, cmd)

    monkeypatch.setattr(build, "up_to_date", lambda: False)
    monkeypatch.setattr(build, "native_up_to_date", lambda: False)
    monkeypatch.setattr(build.subprocess, "run", run)
    monkeypatch.setattr(build.os, "replace", lambda a, b: None)
    monkeypatch.setattr(build, "nvcc_path", lambda: "/opt/cuda/bin/nvcc")
    return seen


def test_the_library_is_built_where_the_extension_module_cannot_be(commands, capsys):
    assert build.build(force=True) == build.LIB
    assert [os.path.basename(c[0]) for c in commands][0] == "nvcc"
    assert "ctypes" in capsys.readouterr().err


def test_a_library_that_cannot_be_built_is_an_error(commands, monkeypatch):
    def missing():
        raise RuntimeError("nvcc not found")

    monkeypatch.setattr(build, "nvcc_path", missing)
    with pytest.raises(RuntimeError):
        build.build()


def test_the_library_alone_needs_no_c_compiler(commands):
    assert build.build_library() == build.LIB
    assert [os.path.basename(c[0]) for c in commands] == ["nvcc"]
