"""The build on machines that lack something: the C library needs nvcc alone, the binding's native calls are optional."""
import os
import subprocess
import sys

import pytest

from paper_2607_15810_b200 import build as Bd


@pytest.fixture
def built(monkeypatch, tmp_path):
    """build() with the library's compilation recorded instead of run, and _native.so in a folder of the test's."""
    calls = []
    monkeypatch.setattr(Bd, "_build_lib", lambda verbose: calls.append("lib"))
    monkeypatch.setattr(Bd, "NATIVE", str(tmp_path / "_native.so"))
    (tmp_path / "_native.so").write_bytes(b"of older sources")
    return calls


def _built_without_native(calls, capsys):
    assert Bd.build(force=True) == Bd.LIB and calls == ["lib"]
    assert not os.path.exists(Bd.NATIVE)
    assert "_native.so is not built" in capsys.readouterr().err


def test_library_is_built_without_torch(built, monkeypatch, capsys):
    monkeypatch.setitem(sys.modules, "torch", None)                       # (import torch raises ImportError)
    _built_without_native(built, capsys)


def test_library_is_built_without_a_host_compiler(built, monkeypatch, capsys):
    def popen(cmd, **kw):
        raise FileNotFoundError(2, "No such file or directory", cmd[0])
    monkeypatch.setattr(subprocess, "Popen", popen)
    _built_without_native(built, capsys)


def test_library_is_built_where_the_native_calls_do_not_compile(built, monkeypatch, capsys, tmp_path):
    broken = tmp_path / "native.cpp"
    broken.write_text("#include <no_such_header.h>\n")
    monkeypatch.setattr(Bd, "NATIVE_SOURCE", str(broken))
    monkeypatch.setattr(Bd, "CSRC", str(tmp_path))
    _built_without_native(built, capsys)


def test_native_calls_of_another_torch_are_rebuilt(monkeypatch, tmp_path):
    """Newer than its sources is not enough."""
    monkeypatch.setattr(Bd, "NATIVE", str(tmp_path / "_native.so"))
    monkeypatch.setattr(Bd, "needs_build", lambda: False)
    started = []
    monkeypatch.setattr(Bd, "_start_native", lambda: started.append(Bd.native_tag()))
    for tag, times in ((Bd.native_tag(), 0), ("torch 1.0, CUDA 9.0, cxx11 ABI 0, cpython-36m", 1), (Bd.native_tag() + "0", 2)):
        (tmp_path / "_native.so").write_bytes(b"\x7fELF built for " + tag.encode() + b"\0")
        Bd.build()
        assert len(started) == times, tag


def test_native_calls_of_another_torch_are_not_loaded(monkeypatch):
    from paper_2607_15810_b200 import binding as B
    if not os.path.exists(Bd.NATIVE):
        pytest.skip("_native.so is not built here")
    assert Bd.native_matches() and B._native is not None
    monkeypatch.setattr(Bd, "native_tag", lambda: "torch 1.0, CUDA 9.0, cxx11 ABI 0, cpython-36m")
    with pytest.warns(UserWarning, match="_native.so is left out"):
        assert B._load_native() is None
