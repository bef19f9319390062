"""The argument-converting extension is optional: where it cannot be built, or belongs to another header, the binding uses
ctypes (no GPU)."""
import subprocess

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


def test_an_extension_of_another_header_is_not_used(monkeypatch):
    build.build()
    lib = binding.library()
    assert type(binding._load_calls(lib)).__name__ == "module"
    monkeypatch.setattr(build, "abi_fingerprint", lambda: "0" * 16)
    assert isinstance(binding._load_calls(lib), binding._CtypesCalls)


def test_fingerprint_sees_declarations_and_not_comments(monkeypatch, tmp_path):
    text = open(build.INCLUDE + "/svip.h").read()
    here = build.abi_fingerprint()
    monkeypatch.setattr(build, "INCLUDE", str(tmp_path))
    (tmp_path / "svip.h").write_text(text.replace("/*", "/* more words\n", 1))
    assert build.abi_fingerprint() == here
    (tmp_path / "svip.h").write_text(text.replace("int top_k, float top_p", "float top_p, int top_k", 1))
    assert build.abi_fingerprint() != here
