"""What is compiled where: the CUDA library with nvcc alone, the binding's native part only beside a CUDA build of torch, and
again when that is another one.  The compilers are stand-ins that write their output files."""
import types

import pytest

from paper_2104_08378_b200 import build


@pytest.fixture
def compile_(monkeypatch, tmp_path):
    """compile_(torch version or None, with CUDA): the compilers that build_library() calls, in order."""
    monkeypatch.setattr(build, "LIB_PATH", str(tmp_path / "libsp24.so"))
    monkeypatch.setattr(build, "NATIVE_PATH", str(tmp_path / "_native.so"))
    monkeypatch.setattr(build, "NATIVE_STAMP", str(tmp_path / "_native.torch"))
    called = []

    def compiler(command):
        called.append("g++" if command[0] == "g++" else "link" if "--shared" in command else "nvcc")
        open(command[command.index("-o") + 1], "w").close()
    monkeypatch.setattr(build.subprocess, "check_call", compiler)

    def run(version, cuda, **kwargs):
        folder = tmp_path / "torch"
        (folder / "lib").mkdir(parents=True, exist_ok=True)
        (folder / "lib" / "libc10_cuda.so").unlink(missing_ok=True)
        if cuda:
            (folder / "lib" / "libc10_cuda.so").touch()
        spec = types.SimpleNamespace(origin=str(folder / "__init__.py")) if version else None
        monkeypatch.setattr(build.importlib.util, "find_spec", lambda name: spec)
        monkeypatch.setattr(build.importlib.metadata, "version", lambda name: version)
        called.clear()
        needed = build.needs_build()
        build.build_library(**kwargs)
        assert needed == bool(called) or kwargs
        return list(called)
    return run


LIBRARY = ["nvcc"] * len(build.SOURCES) + ["link"]


@pytest.mark.parametrize("version", [None, "2.0+cpu"])
def test_without_a_cuda_build_of_torch(compile_, version):
    assert compile_(version, False) == LIBRARY
    assert compile_(version, False) == []
    assert compile_(version, False, force=True) == LIBRARY


def test_another_torch(compile_):
    assert compile_("2.0+cu1", True) == LIBRARY + ["g++"]
    assert compile_("2.0+cu1", True) == []
    assert compile_("2.1+cu1", True) == ["g++"]
    assert compile_("2.1+cu1", True) == []
    assert compile_("2.1+cu1", True, force=True) == LIBRARY + ["g++"]
