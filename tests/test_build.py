"""What is built without what: the library needs nvcc alone, the extension module a C compiler and Python's headers."""
import os
import sysconfig

import pytest

from paper_2409_13761_b200 import build, kdn


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


@pytest.mark.skipif(kdn._native is None, reason="no C compiler or no Python headers")
def test_a_module_made_from_another_header_or_for_another_interpreter_is_not_used(monkeypatch, tmp_path):
    assert build.NATIVE.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    assert kdn._native.stamp == build.native_stamp()

    def fails(force=False):
        raise RuntimeError("no C compiler found")

    monkeypatch.setattr(build, "build_native", fails)
    with open(build.NATIVE, "rb") as f:
        module = f.read()
    other = tmp_path / os.path.basename(build.NATIVE)
    monkeypatch.setattr(build, "NATIVE", str(other))
    assert kdn._load_native() is None                        # there is none for this interpreter
    other.write_bytes(module)
    assert kdn._load_native().stamp == build.native_stamp()
    other.unlink()
    stamp = build.native_stamp().encode()
    other.write_bytes(module.replace(stamp, stamp[:-1] + (b"0" if stamp[-1:] != b"0" else b"1")))
    os.utime(other, (4e9, 4e9))                              # newer than its source
    assert not build.native_up_to_date() and kdn._load_native() is None
