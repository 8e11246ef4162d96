"""What the build leaves behind where the native marshaller cannot be compiled (no GPU needed)."""
import pytest

from paper_2603_06738_b200 import build


@pytest.mark.parametrize("compiler", ["false", "no-such-compiler"])
def test_the_library_is_built_without_a_compiler_for_the_marshaller(monkeypatch, tmp_path, compiler):
    """nvcc alone builds the library: a marshaller that does not compile leaves a warning, and none of an earlier build."""
    old = tmp_path / "_rib_marshal.so"
    old.write_bytes(b"of an earlier build")
    monkeypatch.setattr(build, "MARSHAL", old)
    monkeypatch.setattr(build, "LIB", tmp_path / "lib.so")
    monkeypatch.setattr(build, "sources", lambda: [])         # nothing to compile: what is asked is the order
    monkeypatch.setattr(build, "PKG", tmp_path)
    monkeypatch.setenv("NVCC", str(tmp_path / "nvcc"))
    nvcc = tmp_path / "nvcc"
    nvcc.write_text('#!/bin/sh\nfor a; do last=$a; done\necho linked > "$last"\n')
    nvcc.chmod(0o755)
    monkeypatch.setenv("CXX", compiler)
    with pytest.warns(RuntimeWarning, match="marshal"):
        lib = build.build(force=True)
    assert lib.read_text() == "linked\n"
    assert not old.exists()
