"""The argument-converting extension is optional: where it cannot be built, or belongs to another header, the binding uses
ctypes (no GPU)."""
import subprocess

import pytest

from paper_2411_18462_b200 import binding, build


def test_a_failing_compiler_leaves_no_extension_and_raises_nothing(monkeypatch, tmp_path, capsys):
    stale = tmp_path / "native_calls.so"
    stale.write_bytes(b"of other sources")
    monkeypatch.setattr(build, "NATIVE", str(stale))

    def fails(cmd, *a, **k):
        raise subprocess.CalledProcessError(1, cmd)
    monkeypatch.setattr(build.subprocess, "check_call", fails)
    assert build.build_native(force=True) is None
    assert not stale.exists() and "ctypes" in capsys.readouterr().err
